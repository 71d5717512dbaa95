"""GPU parity at the edges of the kernels' tiles and dispatch rules: the checks (and their bounds) are those of
test_gpu_parity.py, the cases are the sizes where a tile is ragged, a tile holds several images, or a variant begins or ends."""

import numpy as np
import pytest

import test_gpu_parity as parity

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# N, n_ci, n_co, H, W, P_ci, P_co, P_0, P_1, k
CONVG_EDGES = [
    (7, 2, 9, 14, 14, 1, 1, 2, 2, 5),        # 7 x 7 shards, several images a tile, the last tile of images partly empty; 9 = 5 + 4 channels
    (19, 3, 7, 9, 17, 1, 1, 1, 1, 3),        # odd rows; 7 channels: four pairs, the last half empty
    (5, 1, 1, 3, 3, 1, 1, 1, 1, 7),          # a kernel wider than the image, one channel each way
    (2, 9, 3, 18, 40, 2, 1, 1, 1, 7),        # 16-float windows, uneven input blocks (5, 4)
    (1, 2, 17, 33, 129, 1, 2, 1, 1, 5),      # 9 and 8 channels: groups of 5, 4 and 8; one cell past tile edges
    (3, 6, 5, 20, 31, 1, 1, 3, 1, 3),        # uneven rows (7, 7, 6) beside odd columns
    (4, 2, 8, 301, 310, 1, 1, 1, 1, 3),      # tiles enough for several waves: eight pixels a thread, all of four pairs / one pair
    (300, 4, 7, 30, 39, 1, 1, 1, 1, 5),      # the same with tiles of several images; rows that end inside a thread's pixels
    (200, 4, 10, 29, 31, 1, 2, 1, 1, 7),     # the same, 7 x 7 and two blocks of channels
    (2, 70, 66, 24, 33, 2, 2, 1, 1, 3),      # 90 pairs of channel groups: slices chosen by the turns they make
]


@pytest.mark.parametrize("case", CONVG_EDGES, ids=[str(c) for c in CONVG_EDGES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_generalized_conv_tiles(case, integer):
    parity.test_generalized_conv_fwd_and_adj(case, integer)
    parity.test_generalized_conv_param_gradients(case, integer)


@pytest.mark.parametrize("case", [(104, 112, 640, 5), (16, 16, 1600, 3), (24, 20, 900, 7)], ids=str)
def test_generalized_conv_gradient_sums_stay_short(case):
    """Sums over many pixels are added up in short runs.  dy = 1 + 2^-12 and x = 1: a run of up to 4096 terms is exact in fp32,
    longer ones lose the 2^-12 of every further term; adding up the runs (pair halves, splits, folds, slices: fewer than 100
    additions on a path) costs at most 100 * 2^-24."""
    torch, distdl, dev = parity.torch, parity.distdl, parity.DEV
    ci, co, n, k = case
    h = k // 2
    part = distdl.Partition((1, ci, n, n), (1, 1, 1, 1), (0, 0, h, h), (0, 0, h, h))
    x = torch.ones(part.padded_shape(0), device=dev)
    dy = torch.full((1, co, n, n), 1 + 2.0 ** -12, device=dev)
    dw, db = torch.empty(co, ci, k, k, device=dev), torch.empty(co, device=dev)
    ws = torch.empty(distdl.convg_adj_params_workspace(part, co, 1, k, k), dtype=torch.uint8, device=dev)
    distdl.convg_adj_params(part, co, 1, [x], [dy], (k, k), [dw], [db], ws)
    distdl.device_status()
    cells = n - (torch.arange(k, device=dev, dtype=torch.float64) - h).abs()           # pixels that have the tap inside the tensor
    want = (1 + 2.0 ** -12) * cells[:, None] * cells[None, :]
    assert ((dw.double() - want).abs() <= 100 * 2.0 ** -24 * want).all()
    assert ((db.double() - (1 + 2.0 ** -12) * n * n).abs() <= 100 * 2.0 ** -24 * n * n).all()


@pytest.mark.parametrize("case", [(2, 136, 144, 128, 5), (4, 80, 80, 128, 5), (4, 32, 40, 64, 7)], ids=str)
def test_generalized_conv_gradient_slices_follow_the_device(case):
    """Layers whose pairs of channel groups leave the device far from full, or its last turn far from full, are cut into more
    slices (read off the scratch table: 256 bytes per channel pair and slice), but no more than 16."""
    n, ci, co, side, k = case
    part = parity.distdl.Partition((n, ci, side, side), (1, 1, 1, 1), (0, 0, k // 2, k // 2), (0, 0, k // 2, k // 2))
    slices = parity.distdl.convg_adj_params_workspace(part, co, 1, k, k) / (256 * ci * co)
    assert slices in range(3, 17)


@pytest.mark.parametrize("vector", [16, 32])
@pytest.mark.parametrize("more", [-1, 0, 1, 5, 4097, 70011])
def test_broadcast_around_one_vector_per_resident_thread(vector, more):
    """bfloat16 elements that end anywhere inside a vector, one vector per resident thread (2048 a multiprocessor) and a few less or
    more; the cells around every copy stay untouched."""
    torch = parity.torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * 2048 * vector // 2 + more
    at = 64 if vector == 32 else 8
    src = torch.randint(-2 ** 15, 2 ** 15, (n + at,), device=parity.DEV, dtype=torch.int16)
    bufs = [torch.full((n + at + 64,), 7, device=parity.DEV, dtype=torch.int16) for _ in range(3)]
    parity.distdl.broadcast_fwd(src[at:].view(torch.bfloat16), [b[at:at + n].view(torch.bfloat16) for b in bufs])
    for b in bufs:
        assert torch.equal(b[at:at + n], src[at:]) and (b[:at] == 7).all() and (b[at + n:] == 7).all()


# global NCHW, partition, kernel
CONV_EDGES = [
    ((1, 1, 5, 1), (1, 1, 1, 1), 3),         # one column
    ((1, 1, 6, 1), (1, 1, 1, 1), 3),         # the array ends inside the 16-byte block of the row before the last
    ((1, 1, 7, 1), (1, 1, 1, 1), 5),         # and of the row before that
    ((1, 3, 1, 1), (1, 1, 1, 1), 3),         # of the planes before the last
    ((1, 1, 6, 3), (1, 1, 1, 3), 3),         # the same in three shards
    ((1, 2, 3, 3), (1, 1, 1, 1), 7),         # a kernel wider than the image
    ((1, 2, 9, 66), (1, 1, 1, 1), 7),        # 64-column strips, the last of two columns, narrower than the halo
    ((1, 1, 40, 129), (1, 1, 1, 1), 7),      # 128-column strips, the last of one column
    ((2, 1, 23, 131), (1, 1, 1, 1), 5),      # the last row of a shard ends its array off a 16-byte boundary
    ((1, 2, 50, 516), (1, 1, 1, 3), 5),      # 16-byte rows, strips of 128 and 44 columns
    ((1, 2, 50, 510), (1, 1, 1, 3), 3),      # padded rows (172) on 16-byte boundaries, bulk rows (170) not
    ((1, 1, 30, 408), (1, 1, 1, 3), 7),      # the other way round (142 / 136)
    ((1, 1, 700, 70), (1, 1, 2, 1), 3),      # several row segments per shard
    ((5, 3, 19, 45), (1, 1, 3, 2), 5),       # shards of 7, 6, 6 rows and 23, 22 columns
    ((37, 16, 8, 128), (1, 1, 1, 1), 5),     # strips of 64 columns: as many of 128 as the device has schedulers
    ((37, 16, 9, 128), (1, 1, 1, 1), 5),     # strips of 128: twice as many segments
    # layers that fill the device, in strips of 128 columns (forward, adjoint, gradients: 16-byte reads or not); 250 and 251 columns
    # end the arrays without ghosts off a 16-byte boundary
    ((19, 17, 9, 250), (1, 1, 1, 1), 3),     # 16, not, not
    ((5, 21, 22, 504), (1, 1, 2, 2), 3),     # not, 16, not
    ((19, 17, 9, 251), (1, 1, 1, 1), 5),     # not, not, not
    ((5, 21, 22, 504), (1, 1, 2, 2), 5),     # 16, 16, 16
    ((19, 17, 9, 250), (1, 1, 1, 1), 7),     # 16, not, not
    ((5, 21, 22, 504), (1, 1, 2, 2), 7),     # not, 16, not
]


@pytest.mark.parametrize("case", CONV_EDGES, ids=[str(c) for c in CONV_EDGES])
def test_depthwise_conv_strips(case):
    parity.test_conv_fwd_and_adj(case)
    parity.test_conv_param_gradients(case, True)
    parity.test_conv_param_gradients(case, False)


@pytest.mark.parametrize("width,k", [(64, 3), (128, 3), (128, 5)])
def test_depthwise_conv_gradient_of_an_infinite_cell(width, k):
    """dy = 1 and one infinite cell per channel: the taps that meet the cell inside the tensor are infinite, the others finite, and
    none is NaN, wherever the cell lies among the rows that a warp takes together (3 x 3, and 5 x 5 on 16-byte rows)."""
    torch, distdl, dev = parity.torch, parity.distdl, parity.DEV
    rows, h = 150, k // 2
    at = [0, 1, 2, 3, *range(20, 60), 74, 75, 146, 147, 148, 149]
    part = distdl.Partition((1, len(at), rows, width), (1, 1, 1, 1), (0, 0, h, h), (0, 0, h, h))
    x = torch.ones(part.padded_shape(0), device=dev)
    for c, r in enumerate(at):
        x[0, c, h + r, h + 30] = float("inf")
    dy = torch.ones(1, len(at), rows, width, device=dev)
    dw, db = torch.empty(len(at), k, k, device=dev), torch.empty(len(at), device=dev)
    ws = torch.empty(distdl.conv_adj_params_workspace(part, k, k), dtype=torch.uint8, device=dev)
    distdl.conv_adj_params(part, [x], [dy], (k, k), dw, db, ws)
    distdl.device_status()
    meets = torch.tensor([[0 <= r + h - a < rows for a in range(k)] for r in at], device=dev)
    assert torch.equal(torch.isinf(dw), meets[:, :, None].expand(-1, -1, k)) and not torch.isnan(dw).any()
    assert torch.equal(db, torch.full_like(db, rows * width))


def test_depthwise_conv_host_time_does_not_grow_with_the_image():
    """The cut into row segments is chosen at every call: on shards of 65536 rows in the time of 1024 (a query of the scratch size,
    which chooses it too; best of 30)."""
    import time

    def best(rows):
        part = parity.distdl.Partition((1, 1, rows, 64), (1, 1, 1, 1), (0, 0, 2, 2), (0, 0, 2, 2))
        times = []
        for _ in range(30):
            t = time.perf_counter()
            parity.distdl.conv_adj_params_workspace(part, 5, 5)
            times.append(time.perf_counter() - t)
        return min(times)
    assert best(65536) < best(1024) + 15e-6


# Rows copied chunk by chunk: at least 384 elements, chunks of up to 512, tiles of whole rows in boxes of more than 16384
REPART_EDGES = [
    ((61, 1203), (4, 1), (1, 3)),            # pieces of 401
    ((7, 383 * 3 + 1), (7, 1), (1, 3)),      # pieces of 384 and 383: one each side of the rule; tiles of 256 cut inside a row
    ((200, 383 * 3 + 1), (2, 1), (1, 3)),    # the same in boxes of tiles of whole rows
    ((7, 95 * 3 + 1), (7, 1), (1, 3)),       # short rows: pieces of 96 and 95
    ((300, 1537), (2, 1), (1, 3)),           # pieces of 513 and 512: two chunks and one; several tiles per box
    ((3, 30001), (3, 1), (1, 2)),            # pieces longer than a tile
]
HALO_EDGES = [
    ((40, 403), (2, 2), 1, 1),               # ghost rows of 201 / 202 cells: unit by unit
    ((40, 767), (2, 2), 1, 1),               # of 384 and 383: one each side of the rule
    ((9, 10, 311), (2, 2, 1), (1, 2, 1), (2, 1, 1)),
    ((5, 40001), (2, 1), (1, 0), (1, 0)),
    ((9, 10, 385), (2, 2, 1), (1, 2, 1), (2, 1, 1)),     # rows just long enough to be copied by warps
    ((257, 9, 34), (1, 1, 2), (0, 0, 1), (0, 0, 1)),     # columns of 2313 cells: tiles of 256, the last one of nine
    ((64, 4, 66), (1, 1, 2), (0, 0, 1), (0, 0, 2)),      # 256 cells: one whole tile
]


@pytest.mark.parametrize("case", REPART_EDGES, ids=[str(c) for c in REPART_EDGES])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_repartition_rows(case, dtype):
    parity.test_repartition_fwd_and_adj_bit_exact(case, dtype)


@pytest.mark.parametrize("case", REPART_EDGES, ids=[str(c) for c in REPART_EDGES])
def test_repartition_rows_fp64(case):
    torch, distdl, dev = parity.torch, parity.distdl, parity.DEV
    (rows, cols), src, dst = case
    whole = torch.rand(rows, cols, device=dev, dtype=torch.float64)
    rep = distdl.Repartition((rows, cols), src, dst, distdl.F64)

    def blocks(shapes, axis):
        return [b.clone(memory_format=torch.contiguous_format) for b in torch.split(whole, [s[axis] for s in shapes], axis)]
    rows_of = blocks([rep.shard_shape(w) for w in range(rep.num_src)], 0)
    cols_of = blocks([rep.shard_shape(w, destination=True) for w in range(rep.num_dst)], 1)
    out, back = [torch.empty_like(c) for c in cols_of], [torch.empty_like(r) for r in rows_of]
    distdl.repartition_fwd(rep, rows_of, out)
    distdl.repartition_adj(rep, cols_of, back)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, cols_of)) and all(torch.equal(a, b) for a, b in zip(back, rows_of))


@pytest.mark.parametrize("case", HALO_EDGES, ids=[str(c) for c in HALO_EDGES])
def test_halo_long_rows(case):
    parity.test_halo_fwd_and_adj_bit_exact(case)
    parity.test_halo_fwd_and_adj_bf16_fp64_bit_exact(case)


# nb, nfi, nfo, pfo, pfi: up to 128 samples the weights are the M operand and up to eight blocks share a tile
AFFINE_EDGES = [
    (1, 8, 8, 1, 1),                         # one sample, one partly filled k-block
    (16, 4096, 128, 1, 2),                   # one tile, eight blocks
    (17, 2048, 528, 2, 4),                   # 32 columns for 17 samples, output blocks of 264
    (63, 1000, 136, 1, 1),
    (128, 72, 1032, 3, 1),                   # full batch, a reduction too short to share
    (129, 512, 520, 1, 1),                   # the first batch of the pair variant
]


@pytest.mark.parametrize("case", AFFINE_EDGES, ids=[str(c) for c in AFFINE_EDGES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_affine_few_samples(case, integer):
    parity.test_affine_fwd_and_adj(case, integer)


@pytest.mark.parametrize("case", [(40, 3592, 2048, 1, 1), (70, 7184, 1032, 1, 2)], ids=str)
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_affine_wide_gradient_tiles(case, integer):
    """Tiles enough for 256 columns each; the last one holds eight columns, the last row tile all or eight of its rows."""
    parity.test_affine_param_gradients(case, integer)


@pytest.mark.parametrize("case", [(33, 8, 1040, 2, 1),       # more 64-column groups of db than tiles, the last of eight columns
                                  (9, 16, 72, 1, 1),         # fewer samples than two per warp of db
                                  (300, 1408, 8192, 1, 1)],  # 5 turns of narrow or 3 of wide tiles: wide with five k-blocks, not with four
                         ids=str)
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_affine_bias_gradient_beside_the_tiles(case, integer):
    parity.test_affine_param_gradients(case, integer)


# global shape, partition, kernel, stride, padding
POOL_EDGES = [
    ((1, 1, 7, 5), (1, 1, 1, 1), (3, 3), (1, 1), ((1, 1), (1, 1))),         # every window of a border column is clipped
    ((2, 1, 70, 131), (1, 1, 2, 2), (3, 3), (1, 1), ((1, 1), (1, 1))),
    ((1, 2, 37, 67), (1, 1, 1, 1), (3, 3), (2, 2), ((0, 0), (0, 0))),
    ((1, 1, 300, 22), (1, 1, 2, 1), (2, 2), (2, 2), ((0, 0), (0, 0))),      # several 128-row tiles of warps
    ((1, 3, 9, 260), (1, 1, 1, 2), (3, 3), (2, 2), ((1, 1), (1, 1))),       # 65 outputs: one column past a warp's 64
    ((40, 9, 66, 61), (1, 1, 1, 2), (3, 3), (2, 2), ((1, 1), (1, 1))),      # several rows a warp, every warp at both ends of the rows
    ((90, 16, 75, 33), (1, 1, 1, 1), (3, 3), (1, 1), ((1, 1), (1, 1))),     # 75 rows in equal shares of 16 warps
    ((1, 2, 100, 84), (1, 1, 2, 4), (3, 3), (1, 1), ((1, 1), (1, 1))),      # shards of 21 columns: one column a lane, outputs met on both sides
    ((1, 1, 20, 64), (1, 1, 1, 2), (3, 3), (1, 1), ((1, 1), (1, 1))),       # of 32
    ((1, 1, 20, 66), (1, 1, 2, 2), (3, 3), (1, 1), ((1, 1), (1, 1))),       # of 33: two columns a lane
    ((1, 2, 30, 512), (1, 1, 2, 4), (3, 3), (2, 2), ((1, 1), (1, 1))),      # whole strips, every other row off an 8-byte boundary
    ((1, 1, 61, 259), (1, 1, 3, 2), (2, 2), (2, 2), ((0, 0), (0, 0))),      # windows cut by shards' ends
    ((1, 1, 30, 31), (1, 1, 4, 4), (3, 3), (1, 1), ((0, 0), (0, 0))),       # two columns of a neighbour's outputs: the local adjoint, then H*
    ((1, 1, 6, 7), (1, 1, 3, 3), (3, 3), (2, 2), ((1, 1), (1, 1))),         # one output a shard: the same
    ((8, 60, 264, 36), (1, 1, 1, 2), (3, 3), (2, 2), ((1, 1), (1, 1))),     # 17 rows of groups a warp
    ((1, 2, 20, 20), (1, 1, 2, 4), (2, 2), (2, 2), ((0, 0), (0, 0))),       # a shard that begins with a whole window of the worker on its left
    ((1, 1, 12, 1020), (1, 1, 1, 4), (2, 2), (2, 2), ((0, 0), (0, 0))),     # the same, two groups a lane
    ((1, 1, 24, 75), (1, 1, 5, 5), (2, 2), (2, 2), ((0, 0), (0, 0))),       # on five columns of workers
    ((2, 1, 15, 36), (1, 1, 3, 5), (2, 2), (2, 2), ((0, 1), (0, 1))),       # padded at the end
    ((1, 1, 20, 188), (1, 1, 2, 4), (2, 2), (2, 2), ((1, 1), (1, 1))),      # and at both
    ((1, 1, 9, 257), (1, 1, 1, 2), (3, 3), (2, 2), ((1, 0), (1, 0))),       # 129 columns: the last strip is one, the one before meets the neighbour too
    ((1, 2, 12, 386), (1, 1, 2, 3), (3, 3), (2, 2), ((0, 0), (0, 0))),
    ((1, 1, 10, 514), (1, 1, 1, 4), (3, 3), (2, 2), ((0, 0), (0, 0))),
    ((60, 50, 14, 14), (1, 1, 1, 2), (2, 2), (2, 2), ((0, 0), (0, 0))),     # small images in large batches: the local adjoint, then H*
    ((50, 50, 20, 21), (1, 1, 2, 2), (3, 3), (2, 2), ((1, 1), (1, 1))),
    ((60, 50, 14, 13), (1, 1, 1, 2), (3, 3), (1, 1), ((1, 1), (1, 1))),
]


@pytest.mark.parametrize("case", POOL_EDGES, ids=[str(c[:4]) for c in POOL_EDGES])
@pytest.mark.parametrize("mode", ["avg", "max"])
def test_pool_marching(case, mode):
    parity.test_pool_fwd_and_adj(case, mode)


@pytest.mark.parametrize("stride", [1, 2])
def test_pool_max_of_special_values(stride):
    """NaN, infinities and signed zeros: the first largest cell in window order, a NaN only as the window's first cell."""
    torch, distdl = parity.torch, parity.distdl
    n = 41
    x = np.random.default_rng(5).choice(np.array([np.nan, -np.inf, np.inf, -0.0, 0.0, 1.0, -1.0], dtype=np.float32), size=(n, n))
    w = distdl.halo_widths_1d(n, 1, 3, stride, 1, 1, 1)
    part = distdl.Partition((1, 1, n, n), (1, 1, 1, 1), [0, 0, w[0], w[0]], [0, 0, w[1], w[1]])
    m = (n + 2 - 3) // stride + 1
    pad = np.zeros(part.padded_shape(0), dtype=np.float32)
    pad[0, 0, w[0][0]:w[0][0] + n, w[0][0]:w[0][0] + n] = x
    y, a = torch.empty((1, 1, m, m), device=parity.DEV), torch.empty((1, 1, m, m), dtype=torch.int32, device=parity.DEV)
    distdl.pool_fwd(part, [parity.dev(pad)], (3, 3), (stride, stride), ((1, 1), (1, 1)), distdl.POOL_MAX, [y], [a])
    yr, ar = np.empty((m, m), dtype=np.float32), np.empty((m, m), dtype=np.int32)
    for i in range(m):
        for j in range(m):
            best, where = None, 0
            for k in range(9):
                p, q = i * stride - 1 + k // 3, j * stride - 1 + k % 3
                if 0 <= p < n and 0 <= q < n and (best is None or x[p, q] > best):
                    best, where = x[p, q], k
            yr[i, j], ar[i, j] = best, where
    assert parity.same_bits(parity.host(y)[0, 0], yr) and parity.same_bits(parity.host(a)[0, 0], ar)


# global shape, partition, radius
STENCIL_EDGES = [
    ((3, 3, 3), (1, 1, 1), 4),               # a shard smaller than the radius
    ((1, 1, 5), (1, 1, 1), 1),               # one plane, one row
    ((9, 10, 64), (1, 1, 1), 2),             # whole vectors on one side only: scalar copies in, vectors out, and the other way round
    ((6, 21, 132), (1, 1, 1), 3),            # a second column tile of one vector, a last row tile of five rows
    ((301, 8, 12), (1, 1, 1), 3),            # many chunks of planes, the last one short
    ((10, 17, 258), (2, 2, 2), 4),           # rows 9 and 8, columns 129: shards with different numbers of tiles share the clearing
    ((13, 9, 260), (3, 1, 2), 4),            # planes 5, 4, 4: neighbours exactly as deep as the radius
    ((7, 17, 64), (1, 1, 1), 4),             # tiles of 16 rows x 64 columns, the second of one row
    ((9, 33, 61), (1, 2, 1), 3),             # the same with 4-byte copies, rows 17 and 16
    ((8, 16, 193), (1, 1, 1), 1),            # one column in the last of four tiles
    ((6, 8, 128), (1, 1, 1), 4),             # one tile of 8 rows x 128 columns, two of the others
    ((6, 24, 65), (1, 1, 1), 2),             # 4-byte copies, fewer tiles of 8 x 128
    ((6, 8, 128), (1, 1, 1), 1),             # tiles of 8 x 128 and, in the adjoint, 16-byte copies
    ((9, 8, 256), (1, 1, 2), 2),
    ((11, 24, 200), (2, 3, 1), 3),
]


@pytest.mark.parametrize("case", STENCIL_EDGES, ids=[str(c) for c in STENCIL_EDGES])
def test_stencil_planes_and_rows(case):
    parity.test_stencil3d_fwd_and_adj(case)


@pytest.mark.parametrize("n", [1 << 20, 1000])
@pytest.mark.parametrize("captured", [False, True], ids=["eager", "graph"])
def test_kernels_follow_copies_and_foreign_kernels_in_order(n, captured):
    """Copies, memsets, other libraries' kernels and a second stream between the operators: each sees what came before it."""
    torch, distdl, dev = parity.torch, parity.distdl, parity.DEV
    x = torch.arange(n, device=dev, dtype=torch.float32)
    y, z, w, out = (torch.empty_like(x) for _ in range(4))
    pinned = torch.empty(n, pin_memory=True)
    s, s2 = torch.cuda.Stream(), torch.cuda.Stream()

    def body():
        y.copy_(x)
        distdl.broadcast_fwd(y, [z, w])
        w.zero_()
        distdl.sumreduce_fwd([z, y, w], out)        # 2 x
        out.mul_(2)
        distdl.broadcast_fwd(out, [z])              # 4 x
        pinned.copy_(z, non_blocking=True)
        s2.wait_stream(s)
        with torch.cuda.stream(s2):
            distdl.broadcast_fwd(z, [w])
        s.wait_stream(s2)
        distdl.sumreduce_fwd([w, z], y)             # 8 x

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            body()
        run = graph.replay
    else:
        def run():
            with torch.cuda.stream(s):
                body()
    torch.cuda.synchronize()
    for _ in range(20):
        run()
    torch.cuda.synchronize()
    assert torch.equal(y, 8 * x) and torch.equal(z, 4 * x) and torch.equal(pinned, (4 * x).cpu())


@pytest.mark.parametrize("captured", [False, True], ids=["eager", "graph"])
@pytest.mark.parametrize("op", ["halo_adj", "affine_adj_params"])
def test_operators_of_two_kinds_of_work_see_what_came_before(op, captured):
    """H* with a plan for its row ends, and dW with db: a writer of their inputs, the operator, a reader of its results, with no
    wait of the host between passes and other inputs in each; against the same passes with a wait after every step."""
    torch, distdl, dev = parity.torch, parity.distdl, parity.DEV
    gen = torch.Generator(device=dev)
    gen.manual_seed(3)
    if op == "halo_adj":
        part = distdl.Partition((72, 96, 128), (2, 2, 2), (4,) * 3, (4,) * 3)
        assert part.uses_row_plan(adjoint=True)
        base = [torch.rand(part.padded_shape(w), device=dev, generator=gen) for w in range(8)]
        ins = outs = [torch.empty_like(b) for b in base]
        call = lambda: distdl.halo_adj(part, ins)
    else:
        base = [torch.randn(192, 520, device=dev, generator=gen).bfloat16(), torch.randn(192, 1032, device=dev, generator=gen).bfloat16()]
        ins = [torch.empty_like(b) for b in base]
        outs = [torch.empty(520, 1032, device=dev), torch.empty(520, device=dev)]
        call = lambda: distdl.affine_adj_params(192, 1032, 520, 1, 1, [ins[0]], [ins[1]], [outs[0]], [outs[1]])
    scale = torch.ones((), device=dev)

    def body(wait=lambda: None):
        for i, b in zip(ins, base):
            torch.mul(b, scale, out=i)          # the operator's input, by a kernel of another library
            wait()
        call()
        wait()
        got = [o.clone() for o in outs]
        wait()
        return got

    stream = torch.cuda.Stream()
    want = []
    for n in range(20):
        scale.fill_(n - 7.5)
        want.append(body(torch.cuda.synchronize))
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        body()                                  # kernels loaded before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph() if captured else None
    if captured:
        with torch.cuda.graph(graph, stream=stream):
            held = body()
    torch.cuda.synchronize()
    got = []
    with torch.cuda.stream(stream):
        for n in range(20):
            scale.fill_(n - 7.5)
            if captured:
                graph.replay()
                got.append([h.clone() for h in held])
            else:
                got.append(body())
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert all(torch.equal(p.view(torch.int32), q.view(torch.int32)) for p, q in zip(a, b))


def test_halo_names_the_first_overlapping_pair():
    torch, distdl = parity.torch, parity.distdl
    part = distdl.Partition((12, 40), (3, 2), [1, 1], [1, 1])
    size = [int(np.prod(part.padded_shape(w))) for w in range(6)]
    pool = torch.zeros(6 * 4096, device=parity.DEV)
    at = [5 * 4096, 3 * 4096, 4096, 4 * 4096, 4096 + 4, 0]          # shards 2 and 4 share cells, in no address order
    shards = [pool[a:a + n] for a, n in zip(at, size)]
    for op in (distdl.halo_fwd, distdl.halo_adj):
        with pytest.raises(distdl.DistdlError, match="shards 2 and 4 overlap"):
            op(part, shards)
    shards[4] = pool[2 * 4096:2 * 4096 + size[4]]
    distdl.halo_fwd(part, shards)
    torch.cuda.synchronize()
