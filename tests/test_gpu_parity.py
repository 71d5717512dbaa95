"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle on the same
seeded inputs.  Copies (B, H) and fixed-order sums (R, H*) must be bit-exact; the convolution is
compared within a bound derived from its 25-term fp32 accumulation."""

import numpy as np
import pytest

import oracle
import paper_2006_03108_b200 as distdl
from paper_2006_03108_b200 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def host(t):
    return t.detach().cpu().numpy()


def same_bits(a, b):
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    return a.shape == b.shape and a.tobytes() == b.tobytes()


def make_partitions(case):
    gshape, pshape, hlo, hhi = case
    return oracle.Partition(gshape, pshape, hlo, hhi), distdl.Partition(gshape, pshape, _w(hlo, len(gshape)), _w(hhi, len(gshape)))


def _w(h, rank):
    return [h] * rank if isinstance(h, int) else list(h)


def random_shards(opart, seed, kind="uniform"):
    gen = inputs.uniform_pm1 if kind == "uniform" else inputs.integers
    return [gen(opart.padded_shape(w), seed * 1000 + w) for w in range(opart.num_workers)]


# --------------------------------------------------------------------------
# Broadcast / sum-reduce
# --------------------------------------------------------------------------

@pytest.mark.parametrize("n", [1, 3, 4, 1000, 4099, 1 << 20, (1 << 22) + 5])
@pytest.mark.parametrize("k", [1, 2, 3, 8, 19])
def test_broadcast_bit_exact(n, k):
    x = inputs.uniform_pm1((n,), n + k)
    src = dev(x)
    dsts = [torch.full((n + 8,), 7.0, device=DEV)[:n] for _ in range(k)]
    distdl.broadcast_fwd(src, dsts)
    torch.cuda.synchronize()
    ref = oracle.broadcast_fwd(x, k)
    for d, r in zip(dsts, ref):
        assert same_bits(host(d), r)


def test_broadcast_bf16_and_in_place():
    x = inputs.f32_to_bf16_bits(inputs.normal((12345,), 3))
    src = dev(x.view(np.int16)).view(torch.bfloat16)
    dsts = [src] + [torch.zeros_like(src) for _ in range(3)]
    distdl.broadcast_fwd(src, dsts)
    torch.cuda.synchronize()
    for d in dsts:
        assert same_bits(host(d.view(torch.int16)).view(np.uint16), x)


@pytest.mark.parametrize("shift", [(0, 0), (4, 0), (0, 4), (4, 4)], ids=["32/32", "16/32", "32/16", "16/16"])
def test_broadcast_alignment_paths(shift):
    # source / destinations aligned to 32 bytes take 256-bit accesses, anything else 16-byte ones;
    # the cells around every destination must stay untouched
    n, k = 100003, 3
    x = inputs.uniform_pm1((n,), 17)
    s_off, d_off = shift
    src = torch.zeros(n + 16, device=DEV)
    src[s_off:s_off + n] = dev(x)
    bufs = [torch.full((n + 16,), 7.0, device=DEV) for _ in range(k)]
    distdl.broadcast_fwd(src[s_off:s_off + n], [b[d_off:d_off + n] for b in bufs])
    torch.cuda.synchronize()
    for b in bufs:
        h = host(b)
        assert same_bits(h[d_off:d_off + n], x)
        assert np.all(h[:d_off] == 7.0) and np.all(h[d_off + n:] == 7.0)


@pytest.mark.parametrize("n", [1, 5, 1000, 4099, (1 << 21) + 3])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8, 16, 17, 35])
def test_sumreduce_bit_exact(n, k):
    parts = [inputs.uniform_pm1((n,), 100 * k + i) * np.float32(10.0 ** (i % 5)) for i in range(k)]
    srcs = [dev(p) for p in parts]
    dst = torch.empty(n, device=DEV)
    distdl.sumreduce_fwd(srcs, dst)
    torch.cuda.synchronize()
    assert same_bits(host(dst), oracle.sumreduce_fwd(parts))
    # adjoint names are the same operators
    dst2 = torch.empty(n, device=DEV)
    distdl.broadcast_adj(srcs, dst2)
    torch.cuda.synchronize()
    assert same_bits(host(dst2), host(dst))


def test_sumreduce_signed_zero_and_in_place():
    a = np.array([-0.0, 1e8, 1.0, -0.0, 5.0], dtype=np.float32)
    b = np.array([-0.0, -1e8, 1e8, 0.0, 5.0], dtype=np.float32)
    c = np.array([-0.0, 1.0, -1e8, -0.0, 5.0], dtype=np.float32)
    srcs = [dev(a), dev(b), dev(c)]
    distdl.sumreduce_fwd(srcs, srcs[0])          # dst aliases source 0
    torch.cuda.synchronize()
    assert same_bits(host(srcs[0]), oracle.sumreduce_fwd([a, b, c]))
    one = dev(a)
    out = torch.empty_like(one)
    distdl.sumreduce_fwd([one], out)             # k = 1 keeps -0.0
    torch.cuda.synchronize()
    assert same_bits(host(out), a)


def test_reduce_after_broadcast_and_dot_test():
    k, n = 8, 100003
    x = inputs.uniform_pm1((n,), 7)
    ys = [inputs.uniform_pm1((n,), 70 + i) for i in range(k)]
    copies = [torch.empty(n, device=DEV) for _ in range(k)]
    distdl.broadcast_fwd(dev(x), copies)
    back = torch.empty(n, device=DEV)
    distdl.sumreduce_fwd(copies, back)
    bsy = torch.empty(n, device=DEV)
    distdl.broadcast_adj([dev(y) for y in ys], bsy)
    torch.cuda.synchronize()
    assert same_bits(host(back), oracle.sumreduce_fwd(oracle.broadcast_fwd(x, k)))
    assert np.allclose(host(back), 8 * x, rtol=1e-6, atol=0)
    r = oracle.adjoint_test_ratio([host(c) for c in copies], ys, [x], [host(bsy)])
    assert r < 1e-5


# --------------------------------------------------------------------------
# Broadcast / sum-reduce along partition dimensions
# --------------------------------------------------------------------------

PARTITION_BROADCAST_CASES = [
    # source partition, destination partition, elements per source worker, dtype
    ((1, 4), (4, 4), [256 * 2048] * 4, "f32"),                       # the affine layer's x: 1 x P_fi -> P_fo x P_fi
    ((4, 1), (4, 4), [70001, 3, 4099, 1 << 16], "f32"),              # its y^ -> y: P_fo x P_fi -> P_fo x 1, ragged sizes
    ((1, 1, 2, 2, 2), (1, 3, 2, 2, 2), [5000 + 7 * i for i in range(8)], "f32"),   # the convolution's x: ... -> 1 x P_co x P_ci x P_0 x P_1
    ((1, 2, 1, 2, 2), (1, 2, 3, 2, 2), [4096] * 8, "bf16"),          # its y: 1 x P_co x 1 x P_0 x P_1 <- 1 x P_co x P_ci x P_0 x P_1
    ((1,), (20,), [33333], "f64"),                                   # more copies than one launch takes
    ((3,), (3,), [100, 200, 300], "f32"),                            # equal partitions
]


@pytest.mark.parametrize("case", PARTITION_BROADCAST_CASES, ids=[str(c[0]) + "->" + str(c[1]) for c in PARTITION_BROADCAST_CASES])
def test_partition_broadcast_and_sumreduce_bit_exact(case):
    src_p, dst_p, sizes, dtype = case
    src_of = oracle.primitives._partition_sources(src_p, dst_p)
    scaled = lambda n, seed: (inputs.uniform_pm1((n,), seed) * np.float32(10.0) ** inputs.integers((n,), seed + 1, -3, 4)).astype(np.float32)
    x32 = [scaled(n, 5000 + 2 * j) for j, n in enumerate(sizes)]
    y32 = [scaled(sizes[j], 6000 + 2 * w) for w, j in enumerate(src_of)]
    if dtype == "bf16":
        x, y = [inputs.f32_to_bf16_bits(a) for a in x32], [inputs.f32_to_bf16_bits(a) for a in y32]
        up, back, add = _bits_dev, _bits_host, oracle.bf16_add
        empty = lambda n: torch.empty(n, dtype=torch.bfloat16, device=DEV)
    elif dtype == "f64":
        x, y = [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in x32], [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in y32]
        up, back, add = dev, host, None
        empty = lambda n: torch.empty(n, dtype=torch.float64, device=DEV)
    else:
        x, y, up, back, add = x32, y32, dev, host, None
        empty = lambda n: torch.empty(n, device=DEV)
    xs, ys = [up(a) for a in x], [up(a) for a in y]
    out = [empty(sizes[j]) for j in src_of]
    distdl.partition_broadcast_fwd(src_p, dst_p, xs, out)
    dx = [empty(n) for n in sizes]
    distdl.partition_broadcast_adj(src_p, dst_p, ys, dx)
    torch.cuda.synchronize()
    for got, ref in zip(out, oracle.partition_broadcast_fwd(src_p, dst_p, x)):
        assert same_bits(back(got), ref)
    for got, ref in zip(dx, oracle.partition_broadcast_adj(src_p, dst_p, y, add=add)):
        assert same_bits(back(got), ref)
    if dtype == "f32":
        r = oracle.adjoint_test_ratio([host(t) for t in out], y, x, [host(t) for t in dx])
        assert r < 1e-5


# --------------------------------------------------------------------------
# Halo exchange
# --------------------------------------------------------------------------

HALO_CASES = [
    ((11,), (3,), 2, 2),
    ((7,), (1,), 1, 2),
    ((10,), (4,), [[0, 1, 2, 1]], [[1, 0, 2, 0]]),
    ((6, 6), (2, 2), 1, 1),
    ((7, 5), (3, 2), (1, 2), (2, 1)),
    ((9, 8), (2, 2), [[0, 4], [3, 0]], [[2, 0], [0, 3]]),
    ((9, 8), (2, 2), [[0, 4], [0, 3]], [[2, 0], [0, 0]]),      # Appendix B.2 widths
    ((5, 6, 7), (2, 1, 3), (1, 2, 1), (1, 0, 2)),
    ((4, 4, 4), (2, 2, 2), 1, 1),
    ((6, 4), (3, 1), 2, 2),                                   # thin: a cell receives from both sides
    ((3, 3, 3), (3, 3, 3), 1, 1),                             # 27 sources per cell
    ((3, 3, 2, 4), (1, 1, 2, 2), (0, 0, 1, 1), (0, 0, 1, 1)),
    ((4, 5, 6, 4, 6), (2, 1, 2, 1, 2), (1, 0, 1, 1, 2), (0, 1, 1, 0, 1)),
    ((256, 256), (2, 2), 1, 1),                               # the small 2-D configuration
    ((70, 66, 72), (2, 2, 2), 4, 4),                          # 16-byte paths, several tiles
    ((67, 61, 68), (3, 2, 2), (2, 4, 4), (3, 4, 4)),          # uneven split, mixed alignment
    ((2, 3, 40, 44), (1, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2)),
]

# Geometries whose innermost dimension is made of whole 16-byte units (fp32: multiples of 4): these run through
# the row plan (ghost rows written end to end, the ghosts at the row ends staged through shared memory).
ROW_PLAN_CASES = [
    ((40,), (2,), 4, 4),                                      # rank 1: row ends only
    ((12, 16), (3, 1), (1, 4), (1, 4)),                       # one worker along the rows: both row ends are cleared
    ((13, 48), (3, 2), (1, 4), (2, 8)),                       # uneven rows, different widths per side
    ((9, 7, 64), (2, 3, 4), [[1, 2], [0, 1, 2], [4, 0, 8, 4]], [[2, 0], [1, 1, 0], [4, 8, 0, 4]]),   # per-worker widths
    ((10, 10, 72), (3, 2, 3), (1, 2, 4), (2, 1, 4)),          # uneven outer splits
    ((3, 3, 6, 16), (1, 1, 2, 2), (0, 0, 1, 4), (0, 0, 1, 4)),
    ((4, 5, 6, 4, 16), (2, 1, 2, 1, 2), (1, 0, 1, 1, 4), (0, 1, 1, 0, 4)),
    ((150, 40, 136), (2, 2, 2), (3, 2, 8), (1, 4, 4)),        # several blocks per worker, two units per ghost
    ((64, 48), (4, 4), (2, 0), (2, 0)),                       # no ghosts along the rows: row blocks only
    ((8, 8, 1040), (2, 2, 2), (1, 1, 260), (1, 1, 260)),      # ghosts half as wide as the bulk
]
HALO_CASES += ROW_PLAN_CASES


def test_row_plan_is_used_where_the_geometry_allows_it():
    for case in ROW_PLAN_CASES + [((70, 66, 72), (2, 2, 2), 4, 4)]:
        assert make_partitions(case)[1].uses_row_plan(), case
    for case in [((11,), (3,), 2, 2), ((67, 61, 68), (3, 2, 2), (2, 4, 4), (3, 4, 4)), ((256, 256), (2, 2), 1, 1)]:
        assert not make_partitions(case)[1].uses_row_plan(), case


@pytest.mark.parametrize("case", HALO_CASES, ids=[str(c[0]) + str(c[1]) for c in HALO_CASES])
def test_halo_fwd_and_adj_bit_exact(case):
    opart, gpart = make_partitions(case)
    for w in range(opart.num_workers):
        assert gpart.padded_shape(w) == opart.padded_shape(w)
    x = random_shards(opart, 11)                         # ghosts hold garbage on entry
    xs = [dev(a) for a in x]
    distdl.halo_fwd(gpart, xs)
    torch.cuda.synchronize()
    ref = oracle.halo_fwd_sequence(opart, x)
    for w in range(opart.num_workers):
        assert same_bits(host(xs[w]), ref[w]), "H differs on worker %d" % w
    y = random_shards(opart, 12)
    ys = [dev(a) for a in y]
    distdl.halo_adj(gpart, ys)
    torch.cuda.synchronize()
    refa = oracle.halo_adj_sequence(opart, y)
    for w in range(opart.num_workers):
        assert same_bits(host(ys[w]), refa[w]), "H* differs on worker %d" % w
    # the adjoint (dot-product) test on the GPU results, fp64 inner products over every cell
    r = oracle.adjoint_test_ratio([host(t) for t in xs], y, x, [host(t) for t in ys])
    assert r < 1e-5


def test_bounded_wait_runs_out_and_reports_timeout():
    """A wait that nothing ends: the kernel gives up after its limit (here about a millisecond of SM cycles),
    returns by itself and leaves DISTDL_ERR_TIMEOUT in the status word, once; the context stays usable."""
    distdl.device_status()
    distdl.selftest_wait_timeout(2_000_000)
    with pytest.raises(distdl.DistdlError) as err:
        distdl.device_status()
    assert err.value.status == 6 and "wait" in str(err.value)
    distdl.device_status()                                   # reported once, then clear again
    x = inputs.uniform_pm1((4097,), 77)
    out = [torch.empty(4097, device=DEV) for _ in range(2)]
    distdl.broadcast_fwd(dev(x), out)                        # ordinary work still runs
    torch.cuda.synchronize()
    assert all(same_bits(host(o), x) for o in out)
    with pytest.raises(distdl.DistdlError):
        distdl.selftest_wait_timeout(10 ** 12)               # limits of seconds are refused


def test_halo_adj_order_sensitive_values():
    """Values of very different magnitude: any other summation order changes the bits."""
    case = ((12, 12, 12), (2, 2, 2), 2, 2)
    opart, gpart = make_partitions(case)
    y = []
    for w in range(opart.num_workers):
        a = inputs.uniform_pm1(opart.padded_shape(w), 900 + w)
        scale = np.float32(10.0) ** inputs.integers(opart.padded_shape(w), 950 + w, -6, 7)
        y.append((a * scale).astype(np.float32))
    ys = [dev(a) for a in y]
    distdl.halo_adj(gpart, ys)
    torch.cuda.synchronize()
    ref = oracle.halo_adj_sequence(opart, y)
    for w in range(opart.num_workers):
        assert same_bits(host(ys[w]), ref[w])


def test_halo_bf16_copies():
    case = ((20, 24), (2, 2), 2, 2)
    opart = oracle.Partition(*case)
    gpart = distdl.Partition(case[0], case[1], [2, 2], [2, 2], dtype=distdl.BF16)
    x = [inputs.f32_to_bf16_bits(a) for a in random_shards(opart, 13)]
    xs = [dev(a.view(np.int16)).view(torch.bfloat16) for a in x]
    distdl.halo_fwd(gpart, xs)
    torch.cuda.synchronize()
    ref = oracle.halo_fwd_definition(opart, x)            # copies of bit patterns
    for w in range(opart.num_workers):
        assert same_bits(host(xs[w].view(torch.int16)).view(np.uint16), ref[w])


def test_operator_calls_replay_from_a_cuda_graph():
    """The calls only enqueue kernels on the given stream, so a captured sequence replays with the same bits."""
    case = ((70, 66, 72), (2, 2, 2), 4, 4)
    opart, gpart = make_partitions(case)
    x, y = random_shards(opart, 41), random_shards(opart, 42)
    xs, ys = [dev(a) for a in x], [dev(a) for a in y]
    srcs = [dev(inputs.uniform_pm1((5000,), 4300 + i)) for i in range(3)]
    red = torch.empty(5000, device=DEV)
    # first calls outside the capture (one-time set-up of kernel attributes happens on first use)
    distdl.halo_fwd(gpart, [t.clone() for t in xs])
    distdl.halo_adj(gpart, [t.clone() for t in ys])
    distdl.sumreduce_fwd(srcs, red)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            distdl.halo_fwd(gpart, xs)
            distdl.halo_adj(gpart, ys)
            distdl.sumreduce_fwd(srcs, red)
    for t, a in zip(xs + ys, x + y):                 # capture does not run anything: restore and replay
        t.copy_(dev(a))
    red.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(xs, oracle.halo_fwd_sequence(opart, x)):
        assert same_bits(host(a), b)
    for a, b in zip(ys, oracle.halo_adj_sequence(opart, y)):
        assert same_bits(host(a), b)
    assert same_bits(host(red), oracle.sumreduce_fwd([host(t) for t in srcs]))


# --------------------------------------------------------------------------
# bfloat16 and fp64 variants of B, R, H, H*, all-reduce
# --------------------------------------------------------------------------

def _bits_dev(bits):
    return dev(np.ascontiguousarray(bits).view(np.int16)).view(torch.bfloat16)


def _bits_host(t):
    return host(t.view(torch.int16)).view(np.uint16)


@pytest.mark.parametrize("n", [1, 7, 8, 1001, (1 << 20) + 3])
@pytest.mark.parametrize("k", [1, 2, 3, 8, 19])
def test_sumreduce_and_broadcast_bf16_fp64_bit_exact(n, k):
    parts = [inputs.uniform_pm1((n,), 500 * k + i) * np.float32(10.0 ** (i % 5)) for i in range(k)]
    # fp64
    p64 = [p.astype(np.float64) * (1.0 + 2.0 ** -30 * (i + 1)) for i, p in enumerate(parts)]
    dst = torch.empty(n, dtype=torch.float64, device=DEV)
    distdl.sumreduce_fwd([dev(p) for p in p64], dst)
    copies = [torch.empty(n, dtype=torch.float64, device=DEV) for _ in range(k)]
    distdl.broadcast_fwd(dev(p64[0]), copies)
    # bfloat16
    pbf = [inputs.f32_to_bf16_bits(p) for p in parts]
    dstb = torch.empty(n, dtype=torch.bfloat16, device=DEV)
    distdl.sumreduce_fwd([_bits_dev(p) for p in pbf], dstb)
    ar = [_bits_dev(p) for p in pbf]
    distdl.allreduce(ar)
    torch.cuda.synchronize()
    assert same_bits(host(dst), oracle.sumreduce_fwd(p64))
    assert all(same_bits(host(c), p64[0]) for c in copies)
    refb = oracle.sumreduce_fwd(pbf, add=oracle.bf16_add)
    assert same_bits(_bits_host(dstb), refb)
    assert all(same_bits(_bits_host(t), refb) for t in ar)


HALO_DTYPE_CASES = [HALO_CASES[i] for i in (0, 5, 7, 9, 10, 12, 14, 15)]


@pytest.mark.parametrize("case", HALO_DTYPE_CASES, ids=[str(c[0]) + str(c[1]) for c in HALO_DTYPE_CASES])
def test_halo_fwd_and_adj_bf16_fp64_bit_exact(case):
    gshape, pshape, hlo, hhi = case
    opart = oracle.Partition(gshape, pshape, hlo, hhi)
    rank = len(gshape)
    for code in (distdl.F64, distdl.BF16):
        gpart = distdl.Partition(gshape, pshape, _w(hlo, rank), _w(hhi, rank), dtype=code)
        x32, y32 = random_shards(opart, 21), []
        for w in range(opart.num_workers):      # values of very different magnitude: the order of the sums shows in the bits
            a = inputs.uniform_pm1(opart.padded_shape(w), 2200 + w)
            y32.append((a * np.float32(10.0) ** inputs.integers(opart.padded_shape(w), 2300 + w, -3, 4)).astype(np.float32))
        if code == distdl.F64:
            x = [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in x32]
            y = [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in y32]
            xs, ys = [dev(a) for a in x], [dev(a) for a in y]
            add, back = None, host
        else:
            x = [inputs.f32_to_bf16_bits(a) for a in x32]
            y = [inputs.f32_to_bf16_bits(a) for a in y32]
            xs, ys = [_bits_dev(a) for a in x], [_bits_dev(a) for a in y]
            add, back = oracle.bf16_add, _bits_host
        distdl.halo_fwd(gpart, xs)
        distdl.halo_adj(gpart, ys)
        torch.cuda.synchronize()
        for a, b in zip(xs, oracle.halo_fwd_sequence(opart, x)):
            assert same_bits(back(a), b)
        for a, b in zip(ys, oracle.halo_adj_sequence(opart, y, add=add)):
            assert same_bits(back(a), b)


PERIODIC_HALO_CASES = [
    # global shape, partition, halo lo, halo hi, periodic
    ((7,), (1,), (2,), (3,), (True,)),
    ((9,), (2,), (2,), (1,), (True,)),
    ((6, 8), (2, 2), (1, 1), (2, 2), (True, False)),
    ((12, 16), (1, 3), (2, 1), (1, 2), (True, True)),
    ((8, 10, 12), (2, 1, 2), (1, 1, 1), (1, 1, 1), (False, True, True)),
    ((70, 66, 72), (2, 2, 2), (4, 4, 4), (4, 4, 4), (True, True, True)),      # 16-byte paths, several tiles
    ((16,), (1,), (4,), (8,), (True,)),                                       # a worker that is its own neighbour
    ((12, 32), (1, 2), (2, 4), (1, 8), (True, True)),                         # the same neighbour on both sides
    ((6, 10, 48), (2, 1, 3), (1, 2, 4), (2, 1, 4), (True, False, True)),
]


@pytest.mark.parametrize("case", PERIODIC_HALO_CASES, ids=[str(c[0]) + str(c[1]) + str(c[4]) for c in PERIODIC_HALO_CASES])
def test_periodic_halo_fwd_and_adj_bit_exact(case):
    gs, ps, hlo, hhi, per = case
    opart = oracle.Partition(gs, ps, hlo, hhi, per)
    gpart = distdl.Partition(gs, ps, hlo, hhi, periodic=per)
    x = random_shards(opart, 31)
    xs = [dev(a) for a in x]
    distdl.halo_fwd(gpart, xs)
    y = []
    for w in range(opart.num_workers):
        a = inputs.uniform_pm1(opart.padded_shape(w), 3200 + w)
        y.append((a * np.float32(10.0) ** inputs.integers(opart.padded_shape(w), 3300 + w, -3, 4)).astype(np.float32))
    ys = [dev(a) for a in y]
    distdl.halo_adj(gpart, ys)
    torch.cuda.synchronize()
    for a, b in zip(xs, oracle.halo_fwd_sequence(opart, x)):
        assert same_bits(host(a), b)
    for a, b in zip(ys, oracle.halo_adj_sequence(opart, y)):
        assert same_bits(host(a), b)
    r = oracle.adjoint_test_ratio([host(t) for t in xs], y, x, [host(t) for t in ys])
    assert r < 1e-5


# --------------------------------------------------------------------------
# Convolution layer
# --------------------------------------------------------------------------

CONV_CASES = [
    # global NCHW, partition, kernel
    ((1, 2, 12, 13), (1, 1, 1, 1), 5),
    ((2, 3, 12, 13), (1, 1, 2, 2), 5),
    ((1, 2, 17, 19), (1, 1, 3, 2), 3),
    ((1, 2, 23, 29), (1, 1, 2, 3), 7),
    ((2, 2, 150, 300), (1, 1, 2, 2), 5),     # partial tiles in both directions
    ((1, 3, 140, 264), (1, 1, 2, 2), 5),     # 16-byte aligned rows
    ((1, 2, 130, 520), (1, 1, 1, 2), 3),
    ((1, 1, 64, 1040), (1, 1, 1, 4), 7),
    ((1, 2, 300, 520), (1, 1, 2, 2), 5),     # three strips per shard, vertical neighbours, 16-byte rows
    ((1, 1, 200, 1032), (1, 1, 3, 2), 7),
    ((1, 1, 100, 780), (1, 1, 2, 3), 3),
    ((1, 2, 70, 260), (1, 1, 2, 2), 3),      # padded rows of whole 16-byte units, bulk rows not (K = 3)
    ((1, 1, 70, 260), (1, 1, 2, 2), 7),      # the same for K = 7; the last tile column holds 2 < 3 columns
    ((1, 2, 66, 264), (1, 1, 2, 2), 5),      # the last tile row holds 1 < 2 rows: the tile above it reaches into the halo
    ((1, 1, 68, 260), (1, 1, 2, 2), 7),      # 2 < 3 rows and 2 < 3 columns
    ((1, 2, 70, 272), (1, 1, 2, 2), 5),      # bulk widths of whole groups of eight columns (136), two tile columns of 128 + 8
    ((1, 2, 70, 272), (1, 1, 2, 2), 3),      # the same for the adjoint of K = 3 (rows 8-byte aligned)
    ((1, 1, 70, 528), (1, 1, 2, 2), 7),      # and of K = 7 (264 columns per worker)
    ((1, 41, 160, 384), (1, 1, 1, 3), 5),    # many planes, strips of exactly 128 columns, 16-byte rows
    ((1, 41, 160, 384), (1, 1, 1, 3), 3),    # the same with padded rows (130) off 16-byte boundaries
]


def _abs_bound(opart, x, w):
    """sum |w||x| per output: the scale of the rounding error of the K*K-term fp32 accumulation,
    |fl(sum) - exact| <= K*K * 2^-24 * sum |w||x| to first order."""
    return oracle.conv_fwd(opart, [np.abs(a) for a in x], np.abs(w))


@pytest.mark.parametrize("case", CONV_CASES, ids=[str(c) for c in CONV_CASES])
def test_conv_fwd_and_adj(case):
    gshape, pshape, k = case
    h = k // 2
    hl = (0, 0, h, h)
    opart = oracle.Partition(gshape, pshape, hl, hl)
    obulk = oracle.Partition(gshape, pshape, 0, 0)
    gpart = distdl.Partition(gshape, pshape, hl, hl)
    xg = inputs.normal(gshape, 31)
    w = inputs.normal((gshape[1], k, k), 32, 0.1)
    bias = inputs.normal((gshape[1],), 33)
    x = oracle.scatter_global(opart, xg, fill=lambda wk: np.full(opart.padded_shape(wk), 1e30, dtype=np.float32))
    xs = [dev(a) for a in x]
    ys = [torch.full(obulk.padded_shape(wk), -7.0, device=DEV) for wk in range(opart.num_workers)]
    distdl.conv_fwd(gpart, xs, dev(w), dev(bias), ys)
    torch.cuda.synchronize()
    ref = oracle.conv_fwd(opart, x, w, bias)
    bound = _abs_bound(opart, x, w)
    # First-order worst case: K*K FMA roundings, one add of the kernel's two partial sums, the oracle's own rounding
    # to fp32: (K*K + 2) * 2^-24 relative to sum |w||x|.  Asserted: the smaller of that and 1e-6, the relative error
    # the operator is specified to (the largest ratio seen over these cases is 2.6e-7 forward, 2.0e-7 adjoint).
    eps = min((k * k + 2) * 2.0 ** -24, 1e-6)
    worst_fwd = 0.0
    for wk in range(opart.num_workers):
        got = host(ys[wk])
        scale = bound[wk] + np.abs(bias)[None, :, None, None]
        err = np.abs(got.astype(np.float64) - ref[wk])
        assert np.all(err <= eps * scale + 1e-30)
        worst_fwd = max(worst_fwd, float(np.max(err / (scale + 1e-30))))
        assert same_bits(host(xs[wk]), x[wk])            # x, ghosts included, is left untouched
    num = np.sqrt(sum(float(np.sum((host(a).astype(np.float64) - b) ** 2)) for a, b in zip(ys, ref)))
    den = np.sqrt(sum(float(np.sum(b.astype(np.float64) ** 2)) for b in ref))
    assert num / den < 1e-6

    # adjoint
    dyg = inputs.normal(gshape, 34)
    dy = oracle.scatter_global(obulk, dyg)
    dys = [dev(a) for a in dy]
    dxs = [torch.full(opart.padded_shape(wk), 3.0, device=DEV) for wk in range(opart.num_workers)]
    distdl.conv_adj(gpart, dys, dev(w), dxs)
    torch.cuda.synchronize()
    refa = oracle.conv_adj(opart, dy, w)
    bounda = oracle.conv_adj(opart, [np.abs(a) for a in dy], np.abs(w))
    worst_adj = 0.0
    for wk in range(opart.num_workers):
        got = host(dxs[wk])
        err = np.abs(got.astype(np.float64) - refa[wk])
        assert np.all(err <= eps * bounda[wk] + 1e-30)
        worst_adj = max(worst_adj, float(np.max(err / (bounda[wk] + 1e-30))))
        mask = np.ones(opart.padded_shape(wk), dtype=bool)
        mask[opart.bulk_slices(wk)] = False
        assert not got[mask].any()                       # ghosts of dx are zero, as H* leaves them
    # dot-product test of the fused pair (bias is not part of the linear operator)
    y0 = [torch.empty_like(t) for t in ys]
    distdl.conv_fwd(gpart, xs, dev(w), None, y0)
    torch.cuda.synchronize()
    xb = oracle.scatter_global(opart, xg)                # zero ghosts: the inner product is over the bulk
    r = oracle.adjoint_test_ratio([host(t) for t in y0], dy, xb, [host(t) for t in dxs])
    assert r < 1e-5
    # achieved figures, next to the bounds above (shown with pytest -s / -rP)
    print("conv %s: max |err| / sum|w||x| forward %.3g, adjoint %.3g (bound %.3g); 2-norm forward %.3g; dot test %.3g"
          % (case, worst_fwd, worst_adj, eps, num / den, r))


@pytest.mark.parametrize("case", CONV_CASES, ids=[str(c) for c in CONV_CASES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_conv_param_gradients(case, integer):
    gshape, pshape, k = case
    h = k // 2
    hl = (0, 0, h, h)
    opart = oracle.Partition(gshape, pshape, hl, hl)
    obulk = oracle.Partition(gshape, pshape, 0, 0)
    gpart = distdl.Partition(gshape, pshape, hl, hl)
    gen = (lambda shp, seed: inputs.integers(shp, seed, -3, 4)) if integer else inputs.normal
    xg, dyg = gen(gshape, 35), gen(gshape, 36)
    # ghosts hold garbage: the fused exchange must not read them
    x = oracle.scatter_global(opart, xg, fill=lambda wk: np.full(opart.padded_shape(wk), 1e30, dtype=np.float32))
    dy = oracle.scatter_global(obulk, dyg)
    xs, dys = [dev(a) for a in x], [dev(a) for a in dy]
    C = gshape[1]
    dw = torch.full((C, k, k), -5.0, device=DEV)
    db = torch.full((C,), -5.0, device=DEV)
    ws = torch.empty(distdl.conv_adj_params_workspace(gpart, k, k), dtype=torch.uint8, device=DEV)
    for _ in range(2):                                   # twice: the scratch table is reused
        distdl.conv_adj_params(gpart, xs, dys, (k, k), dw, db, ws)
    torch.cuda.synchronize()
    dw_ref, db_ref = oracle.conv_adj_params(opart, x, dy, k, k)
    if integer:
        # |terms| <= 9, fewer than 2^20 of them: every partial sum is an exact integer in fp32, any order
        assert np.array_equal(host(dw), dw_ref) and np.array_equal(host(db), db_ref)
    else:
        # fp32 running sums: the longest chain has 16 terms per tile of the channel (a thread's pair half),
        # then the folds over pair halves, lanes, warps and slices
        tiles = gshape[0] * sum(-(-obulk.padded_shape(wk)[2] // 32) * -(-obulk.padded_shape(wk)[3] // 128)
                                for wk in range(opart.num_workers))
        eps = (16 * tiles + 64) * 2.0 ** -24
        mag_w, mag_b = oracle.conv_adj_params(opart, [np.abs(a) for a in oracle.scatter_global(opart, xg)],
                                              [np.abs(a) for a in dy], k, k)
        assert np.all(np.abs(host(dw).astype(np.float64) - dw_ref) <= eps * mag_w)
        assert np.all(np.abs(host(db).astype(np.float64) - db_ref) <= eps * mag_b)
        assert np.linalg.norm(host(dw).astype(np.float64) - dw_ref) <= 1e-5 * np.linalg.norm(mag_w)
    for wk in range(opart.num_workers):
        assert same_bits(host(xs[wk]), x[wk])
    if not integer:
        # dot test in parameter space, forward through the CUDA layer: <Conv(w, b; x), dy> = <w, dw> + <b, db>
        w = inputs.normal((C, k, k), 37, 0.1)
        bias = inputs.normal((C,), 38)
        ys = [torch.empty(obulk.padded_shape(wk), device=DEV) for wk in range(opart.num_workers)]
        distdl.conv_fwd(gpart, xs, dev(w), dev(bias), ys)
        torch.cuda.synchronize()
        r = oracle.adjoint_test_ratio([host(t) for t in ys], dy, [w, bias], [host(dw), host(db)])
        assert r < 1e-5


# --------------------------------------------------------------------------
# Generalized convolution layer (channel partitions)
# --------------------------------------------------------------------------

CONVG_CASES = [
    # N, n_ci, n_co, H, W, P_ci, P_co, P_0, P_1, k
    (2, 4, 6, 9, 10, 2, 3, 2, 2, 3),
    (1, 5, 3, 8, 7, 2, 2, 1, 2, 5),          # uneven channel blocks, odd channel counts (a group of one)
    (1, 3, 4, 40, 150, 1, 1, 1, 1, 5),       # two tile rows and columns in one shard
    (2, 3, 5, 70, 264, 3, 2, 2, 2, 5),       # 16-byte aligned rows, ragged tiles
    (1, 2, 2, 66, 260, 2, 1, 2, 2, 7),       # short last tile row and column
    (1, 4, 4, 34, 131, 2, 2, 1, 1, 3),
    (1, 2, 3, 40, 264, 1, 2, 1, 2, 7),       # 7 x 7: bulk rows of whole 16-byte units (bulk copies in the adjoint)
    (1, 3, 2, 34, 260, 1, 1, 1, 2, 3),       # 3 x 3: padded rows of whole 16-byte units (bulk copies in the forward)
    (2, 2, 2, 33, 264, 2, 2, 2, 2, 3),       # 3 x 3: bulk copies in the adjoint, short last tile row
]


@pytest.mark.parametrize("case", CONVG_CASES, ids=[str(c) for c in CONVG_CASES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_generalized_conv_fwd_and_adj(case, integer):
    N, nci, nco, H, W, pci, pco, p0, p1, k = case
    h = k // 2
    xpart = oracle.Partition((N, nci, H, W), (1, pci, p0, p1), (0, 0, h, h), (0, 0, h, h))
    ypart = oracle.Partition((N, nco, H, W), (1, pco, p0, p1))
    gpart = distdl.Partition((N, nci, H, W), (1, pci, p0, p1), (0, 0, h, h), (0, 0, h, h))
    gen = (lambda shp, seed, std=1.0: inputs.integers(shp, seed, -2, 3)) if integer else inputs.normal
    xg, wg, bg = gen((N, nci, H, W), 61), gen((nco, nci, k, k), 62, 0.2), gen((nco,), 63)
    dyg = gen((N, nco, H, W), 64)
    cs_i, cz_i = oracle.balanced_split(nco, pco)
    cs_j, cz_j = oracle.balanced_split(nci, pci)
    wb = [np.ascontiguousarray(wg[cs_i[i]:cs_i[i] + cz_i[i], cs_j[j]:cs_j[j] + cz_j[j]]) for i in range(pco) for j in range(pci)]
    bb = [np.ascontiguousarray(bg[cs_i[i]:cs_i[i] + cz_i[i]]) for i in range(pco)]
    x = oracle.scatter_global(xpart, xg, fill=lambda wk: np.full(xpart.padded_shape(wk), 1e30, dtype=np.float32))
    dy = oracle.scatter_global(ypart, dyg)
    xs, dys = [dev(a) for a in x], [dev(a) for a in dy]
    wd = [dev(a) for a in wb]
    ys = [torch.full(ypart.padded_shape(wk), -7.0, device=DEV) for wk in range(ypart.num_workers)]
    dxs = [torch.full(xpart.padded_shape(wk), 3.0, device=DEV) for wk in range(xpart.num_workers)]
    distdl.convg_fwd(gpart, nco, pco, xs, wd, [dev(b) for b in bb], ys)
    distdl.convg_adj(gpart, nco, pco, dys, wd, dxs)
    torch.cuda.synchronize()
    xz = oracle.scatter_global(xpart, xg)
    yref = oracle.convg_fwd(xpart, nco, pco, xz, wb, bb)
    dxref = oracle.convg_adj(xpart, nco, pco, dy, wb)
    for wk in range(xpart.num_workers):
        assert same_bits(host(xs[wk]), x[wk])            # x, ghosts included, is left untouched
        mask = np.ones(xpart.padded_shape(wk), dtype=bool)
        mask[xpart.bulk_slices(wk)] = False
        assert not host(dxs[wk])[mask].any()             # ghosts of dx are zero, as H* leaves them
    if integer:
        # small integers: every product and partial sum is exact in fp32, any order
        for a, b in zip(ys + dxs, yref + dxref):
            assert np.array_equal(host(a), b)
        return
    # n_ci * K * K (adjoint: n_co * K * K) FMA roundings and the oracle's own rounding of its fp64 sum to fp32
    ymag = oracle.convg_fwd(xpart, nco, pco, [np.abs(a) for a in xz], [np.abs(a) for a in wb], [np.abs(b) for b in bb])
    dxmag = oracle.convg_adj(xpart, nco, pco, [np.abs(a) for a in dy], [np.abs(a) for a in wb])
    for got, ref, mag, terms in ((ys, yref, ymag, nci * k * k + 1), (dxs, dxref, dxmag, nco * k * k)):
        for a, b, m in zip(got, ref, mag):
            assert np.all(np.abs(host(a).astype(np.float64) - b) <= (terms + 2) * 2.0 ** -24 * m + 1e-30)
    y0 = [torch.empty_like(t) for t in ys]
    distdl.convg_fwd(gpart, nco, pco, xs, wd, None, y0)
    torch.cuda.synchronize()
    r = oracle.adjoint_test_ratio([host(t) for t in y0], dy, xz, [host(t) for t in dxs])
    assert r < 1e-5


@pytest.mark.parametrize("case", CONVG_CASES, ids=[str(c) for c in CONVG_CASES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_generalized_conv_param_gradients(case, integer):
    N, nci, nco, H, W, pci, pco, p0, p1, k = case
    h = k // 2
    xpart = oracle.Partition((N, nci, H, W), (1, pci, p0, p1), (0, 0, h, h), (0, 0, h, h))
    ypart = oracle.Partition((N, nco, H, W), (1, pco, p0, p1))
    gpart = distdl.Partition((N, nci, H, W), (1, pci, p0, p1), (0, 0, h, h), (0, 0, h, h))
    gen = (lambda shp, seed: inputs.integers(shp, seed, -2, 3)) if integer else inputs.normal
    xg, dyg = gen((N, nci, H, W), 71), gen((N, nco, H, W), 72)
    x = oracle.scatter_global(xpart, xg, fill=lambda wk: np.full(xpart.padded_shape(wk), 1e30, dtype=np.float32))
    dy = oracle.scatter_global(ypart, dyg)
    xs, dys = [dev(a) for a in x], [dev(a) for a in dy]
    _, cz_i = oracle.balanced_split(nco, pco)
    _, cz_j = oracle.balanced_split(nci, pci)
    dw = [torch.full((cz_i[i], cz_j[j], k, k), -5.0, device=DEV) for i in range(pco) for j in range(pci)]
    db = [torch.full((cz_i[i],), -5.0, device=DEV) for i in range(pco)]
    ws = torch.empty(distdl.convg_adj_params_workspace(gpart, nco, pco, k, k), dtype=torch.uint8, device=DEV)
    for _ in range(2):                                   # twice: the scratch table is reused
        distdl.convg_adj_params(gpart, nco, pco, xs, dys, (k, k), dw, db, ws)
    distdl.device_status()
    xz = oracle.scatter_global(xpart, xg)
    dw_ref, db_ref = oracle.convg_adj_params(xpart, nco, pco, xz, dy, k, k)
    if integer:
        for a, b in zip(dw + db, dw_ref + db_ref):
            assert np.array_equal(host(a), b)
        return
    tiles = N * sum(-(-ypart.padded_shape(wk)[2] // 32) * -(-ypart.padded_shape(wk)[3] // 128) for wk in range(p0 * p1))
    eps = (16 * tiles + 64) * 2.0 ** -24
    mag_w, mag_b = oracle.convg_adj_params(xpart, nco, pco, [np.abs(a) for a in xz], [np.abs(a) for a in dy], k, k)
    for a, b, m in zip(dw + db, dw_ref + db_ref, mag_w + mag_b):
        assert np.all(np.abs(host(a).astype(np.float64) - b) <= eps * m)
    # parameter-space dot test through the CUDA forward: <Conv(w, b; x), dy> = <w, dw> + <b, db>
    cs_i, _ = oracle.balanced_split(nco, pco)
    cs_j, _ = oracle.balanced_split(nci, pci)
    wg, bg = inputs.normal((nco, nci, k, k), 73, 0.2), inputs.normal((nco,), 74)
    wb = [np.ascontiguousarray(wg[cs_i[i]:cs_i[i] + cz_i[i], cs_j[j]:cs_j[j] + cz_j[j]]) for i in range(pco) for j in range(pci)]
    bb = [np.ascontiguousarray(bg[cs_i[i]:cs_i[i] + cz_i[i]]) for i in range(pco)]
    ys = [torch.empty(ypart.padded_shape(wk), device=DEV) for wk in range(ypart.num_workers)]
    distdl.convg_fwd(gpart, nco, pco, xs, [dev(a) for a in wb], [dev(b) for b in bb], ys)
    distdl.device_status()
    r = oracle.adjoint_test_ratio([host(t) for t in ys], dy, wb + bb, [host(t) for t in dw + db])
    assert r < 1e-5


# --------------------------------------------------------------------------
# 3-D star-stencil layer
# --------------------------------------------------------------------------

STENCIL_CASES = [
    # global shape, partition, radius
    ((16, 16, 16), (1, 1, 1), 4),
    ((40, 36, 48), (2, 2, 2), 4),         # vector path, every kind of neighbour
    ((20, 19, 150), (2, 2, 2), 2),        # odd row lengths: element-wise path, ragged last vector
    ((70, 20, 264), (1, 2, 2), 4),        # two column tiles per shard, the second one partly empty
    ((130, 17, 40), (2, 1, 1), 1),        # two plane chunks per shard
    ((12, 25, 36), (1, 3, 2), 3),
    ((14, 40, 512), (3, 2, 2), 4),        # uneven plane split (5, 5, 4), full 128-column tiles
    ((11, 21, 260), (2, 2, 2), 4),        # shards of 130 columns: a second tile of two columns
]


@pytest.mark.parametrize("case", STENCIL_CASES, ids=[str(c) for c in STENCIL_CASES])
def test_stencil3d_fwd_and_adj(case):
    gshape, pshape, R = case
    opart = oracle.Partition(gshape, pshape, R, R)
    obulk = oracle.Partition(gshape, pshape, 0, 0)
    gpart = distdl.Partition(gshape, pshape, (R,) * 3, (R,) * 3)
    xg = inputs.normal(gshape, 91)
    w = inputs.normal((3, 2 * R + 1), 92, 0.5)
    x = oracle.scatter_global(opart, xg, fill=lambda wk: np.full(opart.padded_shape(wk), 1e30, dtype=np.float32))
    xs = [dev(a) for a in x]
    ys = [torch.full(obulk.padded_shape(wk), -7.0, device=DEV) for wk in range(opart.num_workers)]
    distdl.stencil3d_fwd(gpart, xs, w, ys)
    torch.cuda.synchronize()
    ref = oracle.stencil3d_fwd(opart, x, w)
    bound = oracle.stencil3d_fwd(opart, [np.abs(a) for a in oracle.scatter_global(opart, xg)], np.abs(w))
    # 6R+3 FMA roundings and the oracle's own rounding of its fp64 sum to fp32
    eps = (6 * R + 3 + 2) * 2.0 ** -24
    for wk in range(opart.num_workers):
        assert np.all(np.abs(host(ys[wk]).astype(np.float64) - ref[wk]) <= eps * bound[wk] + 1e-30)
        assert same_bits(host(xs[wk]), x[wk])            # x, ghosts included, is left untouched
    # adjoint
    dy = oracle.scatter_global(obulk, inputs.normal(gshape, 93))
    dys = [dev(a) for a in dy]
    dxs = [torch.full(opart.padded_shape(wk), 3.0, device=DEV) for wk in range(opart.num_workers)]
    distdl.stencil3d_adj(gpart, dys, w, dxs)
    torch.cuda.synchronize()
    refa = oracle.stencil3d_adj(opart, dy, w)
    bounda = oracle.stencil3d_adj(opart, [np.abs(a) for a in dy], np.abs(w))
    worst_adj = 0.0
    for wk in range(opart.num_workers):
        got = host(dxs[wk])
        err = np.abs(got.astype(np.float64) - refa[wk])
        assert np.all(err <= eps * bounda[wk] + 1e-30)
        worst_adj = max(worst_adj, float(np.max(err / (bounda[wk] + 1e-30))))
        mask = np.ones(opart.padded_shape(wk), dtype=bool)
        mask[opart.bulk_slices(wk)] = False
        assert not got[mask].any()                       # ghosts of dx are zero, as H* leaves them
    xb = oracle.scatter_global(opart, xg)
    r = oracle.adjoint_test_ratio([host(t) for t in ys], dy, xb, [host(t) for t in dxs])
    assert r < 1e-5


# --------------------------------------------------------------------------
# Affine layer
# --------------------------------------------------------------------------

AFFINE_CASES = [
    # nb, nfi, nfo, pfo, pfi
    (16, 256, 256, 2, 2),
    (128, 128, 128, 1, 1),
    (200, 512, 384, 3, 2),       # ragged batch (two row tiles, the second partly empty)
    (256, 1024, 512, 4, 4),
    (77, 256, 1024, 1, 2),
    (300, 768, 256, 2, 1),
    (300, 1024, 1024, 2, 4),     # 256-column tiles, reduction split between two pairs (both directions)
    (520, 512, 768, 3, 2),       # forward splits the reduction, adjoint (three workers) does not
    (40, 200, 136, 1, 1),        # blocks that are not multiples of the 128 / 64 tile sizes (multiples of 8)
    (300, 400, 528, 2, 2),       # ... with pairs of blocks: blocks of 200 and 264 features
    (150, 72, 1032, 3, 1),       # a reduction shorter than two k-blocks; 344-feature output blocks
]


def _affine_inputs(nb, nfi, nfo, pfo, pfi, seed, integer=False):
    if integer:
        xg = inputs.integers((nb, nfi), seed, -3, 4)
        wg = inputs.integers((nfo, nfi), seed + 1, -3, 4)
        dyg = inputs.integers((nb, nfo), seed + 2, -3, 4)
    else:
        xg = inputs.normal((nb, nfi), seed)
        wg = inputs.normal((nfo, nfi), seed + 1, nfi ** -0.5)
        dyg = inputs.normal((nb, nfo), seed + 2)
    xb, wb, dyb = (inputs.f32_to_bf16_bits(a) for a in (xg, wg, dyg))
    xs = np.split(xb, pfi, axis=1)
    ws = [blk for row in np.split(wb, pfo, axis=0) for blk in np.split(row, pfi, axis=1)]
    dys = np.split(dyb, pfo, axis=1)
    return xs, ws, dys


def _bf16_dev(bits):
    return dev(np.ascontiguousarray(bits).view(np.int16)).view(torch.bfloat16)


def _rel_errors(got, ref):
    got = np.concatenate([g.astype(np.float64) for g in got], axis=1)
    ref = np.concatenate([r.astype(np.float64) for r in ref], axis=1)
    return np.max(np.abs(got - ref)) / np.max(np.abs(ref)), np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("case", AFFINE_CASES, ids=[str(c) for c in AFFINE_CASES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_affine_fwd_and_adj(case, integer):
    nb, nfi, nfo, pfo, pfi = case
    xs, ws, dys = _affine_inputs(nb, nfi, nfo, pfo, pfi, 41, integer)
    bias = np.split(inputs.integers((nfo,), 44) if integer else inputs.normal((nfo,), 44), pfo)
    x_d, w_d, dy_d = [_bf16_dev(a) for a in xs], [_bf16_dev(a) for a in ws], [_bf16_dev(a) for a in dys]
    b_d = [dev(b) for b in bias]
    y_d = [torch.full((nb, nfo // pfo), -9.0, device=DEV) for _ in range(pfo)]
    dx_d = [torch.full((nb, nfi // pfi), -9.0, device=DEV) for _ in range(pfi)]
    distdl.affine_fwd(nb, nfi, nfo, pfo, pfi, x_d, w_d, b_d, y_d)
    distdl.affine_adj(nb, nfi, nfo, pfo, pfi, dy_d, w_d, dx_d)
    distdl.device_status()
    xf = [oracle.bf16_bits_to_f64(a) for a in xs]
    wf = [oracle.bf16_bits_to_f64(a) for a in ws]
    dyf = [oracle.bf16_bits_to_f64(a) for a in dys]
    y_ref = oracle.affine_fwd(xf, wf, pfo, pfi, bias)
    dx_ref = oracle.affine_adj(dyf, wf, pfo, pfi)
    y, dx = [host(t) for t in y_d], [host(t) for t in dx_d]
    if integer:
        # small integers: every product and partial sum is exact in fp32, any order
        for a, b in zip(y + dx, y_ref + dx_ref):
            assert np.array_equal(a, b)
    else:
        for got, ref in ((y, y_ref), (dx, dx_ref)):
            emax, el2 = _rel_errors(got, ref)
            assert emax < 2e-2 and el2 < 2e-2          # the stated bound
            assert emax < 1e-4 and el2 < 1e-5          # what fp32 accumulation of exact products gives
        # dot-product test of the pair (no bias: it is not part of the linear operator)
        y0 = [torch.empty_like(t) for t in y_d]
        distdl.affine_fwd(nb, nfi, nfo, pfo, pfi, x_d, w_d, None, y0)
        distdl.device_status()
        r = oracle.adjoint_test_ratio([host(t) for t in y0], dyf, xf, dx)
        assert r < 1e-4


@pytest.mark.parametrize("case", AFFINE_CASES, ids=[str(c) for c in AFFINE_CASES])
@pytest.mark.parametrize("integer", [True, False], ids=["int", "normal"])
def test_affine_param_gradients(case, integer):
    nb, nfi, nfo, pfo, pfi = case
    xs, ws, dys = _affine_inputs(nb, nfi, nfo, pfo, pfi, 45, integer)
    x_d, dy_d = [_bf16_dev(a) for a in xs], [_bf16_dev(a) for a in dys]
    dw_d = [torch.full((nfo // pfo, nfi // pfi), -9.0, device=DEV) for _ in range(pfo * pfi)]
    db_d = [torch.full((nfo // pfo,), -9.0, device=DEV) for _ in range(pfo)]
    distdl.affine_adj_params(nb, nfi, nfo, pfo, pfi, dy_d, x_d, dw_d, db_d)
    distdl.device_status()
    xf = [oracle.bf16_bits_to_f64(a) for a in xs]
    dyf = [oracle.bf16_bits_to_f64(a) for a in dys]
    dw_ref, db_ref = oracle.affine_adj_params(dyf, xf, pfo, pfi)
    dw, db = [host(t) for t in dw_d], [host(t) for t in db_d]
    if integer:
        for a, b in zip(dw + db, dw_ref + db_ref):
            assert np.array_equal(a, b)
    else:
        for got, ref in zip(dw, dw_ref):
            emax, el2 = _rel_errors([got], [ref])
            assert emax < 2e-2 and el2 < 2e-2
            assert emax < 1e-4 and el2 < 1e-5
        emax, el2 = _rel_errors([np.concatenate(db)[None]], [np.concatenate(db_ref)[None]])
        assert emax < 1e-5 and el2 < 1e-5
        # dot test in parameter space, forward through the CUDA layer: <Affine(W, b; x), dy> = <W, dW> + <b, db>
        w_d = [_bf16_dev(a) for a in ws]
        bias = np.split(inputs.normal((nfo,), 46), pfo)
        y_d = [torch.empty((nb, nfo // pfo), device=DEV) for _ in range(pfo)]
        distdl.affine_fwd(nb, nfi, nfo, pfo, pfi, x_d, w_d, [dev(b) for b in bias], y_d)
        distdl.device_status()
        wf = [oracle.bf16_bits_to_f64(a) for a in ws]
        r = oracle.adjoint_test_ratio([host(t) for t in y_d], dyf, wf + bias, dw + db)
        assert r < 1e-4
    # db is optional
    distdl.affine_adj_params(nb, nfi, nfo, pfo, pfi, dy_d, x_d, dw_d, None)
    distdl.device_status()


# --------------------------------------------------------------------------
# Distributed pooling layer (unbalanced halos)
# --------------------------------------------------------------------------

POOL_CASES = [
    # global shape, partition, kernel, stride, padding
    ((2, 3, 11, 10), (1, 1, 3, 2), (2, 2), (2, 2), ((0, 0), (0, 0))),
    ((1, 2, 20, 17), (1, 1, 6, 3), (3, 3), (2, 2), ((1, 1), (1, 1))),
    ((1, 1, 12, 12), (1, 1, 2, 2), (3, 2), (1, 2), ((1, 0), (0, 1))),
    ((1, 1, 1, 20), (1, 1, 1, 6), (1, 2), (1, 2), ((0, 0), (0, 0))),      # Fig. B4
    ((2, 2, 130, 203), (1, 1, 4, 4), (3, 3), (2, 2), ((1, 1), (1, 1))),   # several thread-block tiles, ragged
    ((1, 4, 97, 64), (1, 1, 2, 3), (5, 5), (3, 3), ((2, 2), (2, 2))),
    ((1, 1, 64, 64), (1, 1, 1, 1), (2, 2), (2, 2), ((0, 0), (0, 0))),
]


def _pool_parts(case):
    gs, ps, k, s, pad = case
    opart, geo = oracle.pool_partition(gs, ps, k, s, pad)
    gpart = distdl.Partition(gs, ps, [list(h) for h in opart.hlo], [list(h) for h in opart.hhi])
    return opart, geo, gpart


@pytest.mark.parametrize("case", POOL_CASES, ids=[str(c[:2]) for c in POOL_CASES])
@pytest.mark.parametrize("mode", ["avg", "max"])
def test_pool_fwd_and_adj(case, mode):
    gs, ps, k, s, pad = case
    opart, geo, gpart = _pool_parts(case)
    code = distdl.POOL_AVG if mode == "avg" else distdl.POOL_MAX
    xg = inputs.normal(gs, 61)
    xs = oracle.scatter_global(opart, xg, fill=lambda w: inputs.normal(opart.padded_shape(w), 700 + w))   # garbage ghosts
    ys_ref, arg_ref = oracle.pool_fwd(opart, geo, xs, k, s, pad, mode)
    x_d = [dev(a) for a in xs]
    y_d = [torch.full(tuple(y.shape), -9.0, device=DEV) for y in ys_ref]
    a_d = [torch.full(tuple(y.shape), -1, dtype=torch.int32, device=DEV) for y in ys_ref] if mode == "max" else None
    distdl.pool_fwd(gpart, x_d, k, s, pad, code, y_d, a_d)
    torch.cuda.synchronize()
    # the ghosts of x now hold what H puts there
    for got, ref in zip(x_d, oracle.halo_fwd_definition(opart, xs)):
        assert same_bits(host(got), ref)
    for w, (got, ref) in enumerate(zip(y_d, ys_ref)):
        if mode == "max":
            assert same_bits(host(got), ref)
            assert np.array_equal(host(a_d[w]), arg_ref[w])
        else:
            # fp32 sum of kh*kw terms and one multiplication against the fp64 sum rounded once
            bound = (k[0] * k[1] + 2) * 2.0 ** -24 * np.max(np.abs(xg)) + 1e-30
            assert got.shape == ref.shape and np.max(np.abs(host(got) - ref), initial=0.0) <= bound

    dys = [inputs.normal(y.shape, 800 + w) for w, y in enumerate(ys_ref)]
    dx_ref = oracle.pool_adj(opart, geo, dys, k, s, pad, mode, arg_ref)
    dy_d = [dev(a) for a in dys]
    arg_in = None if mode == "avg" else [dev(a) for a in arg_ref]
    dx_d = [torch.full(tuple(opart.padded_shape(w)), 5.0, device=DEV) for w in range(opart.num_workers)]
    distdl.pool_adj(gpart, dy_d, arg_in, k, s, pad, code, dx_d)
    torch.cuda.synchronize()
    dymax = max([float(np.max(np.abs(d), initial=0.0)) for d in dys])
    terms = ((k[0] + s[0] - 1) // s[0]) * ((k[1] + s[1] - 1) // s[1])      # outputs whose window holds one cell
    for w, (got, ref) in enumerate(zip(dx_d, dx_ref)):
        g = host(got)
        if mode == "max" and terms == 1:
            assert same_bits(g, ref)                                       # pure routing, then the fixed-order H*
        else:
            assert np.max(np.abs(g - ref), initial=0.0) <= 4 * (terms + 2) * 2.0 ** -24 * dymax
        ghosts = g.copy()
        ghosts[opart.bulk_slices(w)] = 0
        assert not ghosts.any()
    if mode == "avg":
        # dot-product test of the pair on the device results (the operator acts on the bulk of x)
        x0 = oracle.scatter_global(opart, xg)
        r = oracle.adjoint_test_ratio([host(t) for t in y_d], dys, x0, [host(t) for t in dx_d])
        assert r < 1e-5


def test_pool_rejects_partitions_with_other_widths():
    gs, ps = (1, 1, 16, 16), (1, 1, 2, 2)
    part = distdl.Partition(gs, ps, [0, 0, 1, 1], [0, 0, 1, 1])
    x = [torch.zeros(tuple(part.padded_shape(w)), device=DEV) for w in range(4)]
    y = [torch.zeros(1, 1, 4, 4, device=DEV) for _ in range(4)]
    with pytest.raises(distdl.DistdlError) as e:
        distdl.pool_fwd(part, x, (2, 2), (2, 2), ((0, 0), (0, 0)), distdl.POOL_AVG, y)
    assert e.value.status == 2          # DISTDL_ERR_SHAPE


# --------------------------------------------------------------------------
# Generalized all-to-all, scatter / gather, all-reduce
# --------------------------------------------------------------------------

REPART_CASES = [
    # global shape, source partition, destination partition
    ((7, 9), (2, 1), (1, 3)),
    ((64, 96), (4, 1), (1, 4)),                  # row blocks -> column blocks ("transpose")
    ((5, 40, 68), (1, 2, 3), (5, 1, 1)),
    ((1000003,), (1,), (7,)),                    # scatter
    ((1000003,), (5,), (1,)),                    # gather
    ((2, 3, 130, 260), (1, 1, 4, 4), (1, 1, 16, 1)),
    ((33, 1025), (3, 5), (3, 5)),                # identity
]


@pytest.mark.parametrize("case", REPART_CASES, ids=[str(c) for c in REPART_CASES])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_repartition_fwd_and_adj_bit_exact(case, dtype):
    gs, sp, dp = case
    osrc, odst = oracle.Partition(gs, sp), oracle.Partition(gs, dp)
    code = distdl.F32 if dtype == "f32" else distdl.BF16
    rep = distdl.Repartition(gs, sp, dp, code)
    if dtype == "f32":
        g = inputs.uniform_pm1(gs, 91)
        up = lambda a: dev(a)
        down = lambda t: host(t)
        empty = lambda shape: torch.full(tuple(shape), 3.0, device=DEV)
    else:
        g = inputs.f32_to_bf16_bits(inputs.uniform_pm1(gs, 91))
        up = lambda a: dev(np.ascontiguousarray(a).view(np.int16)).view(torch.bfloat16)
        down = lambda t: host(t.view(torch.int16)).view(np.uint16)
        empty = lambda shape: torch.full(tuple(shape), 3.0, device=DEV, dtype=torch.bfloat16)
    src = oracle.scatter_global(osrc, g)
    for w in range(rep.num_src):
        assert rep.shard_shape(w) == tuple(src[w].shape)
    ref = oracle.repartition_fwd(osrc, odst, src)
    out = [empty(a.shape) for a in ref]
    distdl.repartition_fwd(rep, [up(a) for a in src], out)
    torch.cuda.synchronize()
    for w, (got, r) in enumerate(zip(out, ref)):
        assert rep.shard_shape(w, destination=True) == tuple(r.shape)
        assert same_bits(down(got), r)
    back = [empty(a.shape) for a in src]
    distdl.repartition_adj(rep, out, back)
    torch.cuda.synchronize()
    for got, r in zip(back, oracle.repartition_adj(osrc, odst, ref)):
        assert same_bits(down(got), r)
    for got, r in zip(back, src):                       # the adjoint of a permutation is its inverse
        assert same_bits(down(got), r)


def test_repartition_rejects_overlapping_buffers():
    rep = distdl.Repartition((8, 8), (2, 1), (1, 2))
    a = torch.zeros(64, device=DEV)
    src = [a[:32].view(4, 8), a[32:].view(4, 8)]
    with pytest.raises(distdl.DistdlError) as e:
        distdl.repartition_fwd(rep, src, [a[:32].view(8, 4), torch.zeros(8, 4, device=DEV)])
    assert e.value.status == 1          # DISTDL_ERR_INVALID_ARG


@pytest.mark.parametrize("k", [1, 2, 5, 8])
def test_allreduce_bit_exact(k):
    n = 100003
    parts = [inputs.uniform_pm1((n,), 300 + i) for i in range(k)]
    bufs = [dev(p) for p in parts]
    distdl.allreduce(bufs)
    torch.cuda.synchronize()
    for got, ref in zip(bufs, oracle.allreduce(parts)):
        assert same_bits(host(got), ref)


# --------------------------------------------------------------------------
# Seeded sweep over random small geometries (uneven splits, thin shards, ragged tiles)
# --------------------------------------------------------------------------

def _random_geometry(rng, rank, max_extent, max_workers, max_halo):
    while True:
        ps = [int(rng.integers(1, max_workers + 1)) for _ in range(rank)]
        if int(np.prod(ps)) > 32:
            continue
        gs = [int(rng.integers(p * (max_halo + 1), max(p * (max_halo + 1) + 1, max_extent))) for p in ps]
        return tuple(gs), tuple(ps)


@pytest.mark.parametrize("seed", range(12))
def test_random_halo_geometries(seed):
    rng = np.random.Generator(np.random.Philox(7000 + seed))
    rank = int(rng.integers(1, 5))
    gs, ps = _random_geometry(rng, rank, 40 if rank < 3 else 18, 4, 3)
    per = tuple(bool(rng.integers(0, 2)) for _ in range(rank)) if seed % 3 == 0 else None
    if per is None:
        # per-worker widths, each no wider than the neighbour's bulk
        sizes = [oracle.balanced_split(gs[k], ps[k])[1] for k in range(rank)]
        hlo = [[int(rng.integers(0, min(3, sizes[k][c - 1]) + 1)) if c > 0 else int(rng.integers(0, 4)) for c in range(ps[k])]
               for k in range(rank)]
        hhi = [[int(rng.integers(0, min(3, sizes[k][c + 1]) + 1)) if c + 1 < ps[k] else int(rng.integers(0, 4))
                for c in range(ps[k])] for k in range(rank)]
        opart = oracle.Partition(gs, ps, hlo, hhi)
        gpart = distdl.Partition(gs, ps, hlo, hhi)
    else:
        h = tuple(int(rng.integers(0, 4)) for _ in range(rank))
        opart = oracle.Partition(gs, ps, h, h, per)
        gpart = distdl.Partition(gs, ps, h, h, periodic=per)
    x, y = random_shards(opart, 50 + seed), random_shards(opart, 80 + seed)
    xs, ys = [dev(a) for a in x], [dev(a) for a in y]
    distdl.halo_fwd(gpart, xs)
    distdl.halo_adj(gpart, ys)
    torch.cuda.synchronize()
    for a, b in zip(xs, oracle.halo_fwd_sequence(opart, x)):
        assert same_bits(host(a), b)
    for a, b in zip(ys, oracle.halo_adj_sequence(opart, y)):
        assert same_bits(host(a), b)


@pytest.mark.parametrize("seed", range(10))
def test_random_row_plan_geometries(seed):
    """Random geometries with rows of whole 16-byte units, in all three element types."""
    rng = np.random.Generator(np.random.Philox(7500 + seed))
    rank = int(rng.integers(1, 5))
    code, per_unit = [(distdl.F32, 4), (distdl.F64, 2), (distdl.BF16, 8)][seed % 3]
    gs, ps = _random_geometry(rng, rank, 30 if rank < 3 else 14, 4, 3)
    gs, ps = list(gs), list(ps)
    gs[-1] = ps[-1] * per_unit * int(rng.integers(1, 4))                  # equal blocks of whole units along the rows
    periodic = tuple(bool(rng.integers(0, 2)) for _ in range(rank)) if seed % 2 == 0 else None
    if periodic is None:
        sizes = [oracle.balanced_split(gs[k], ps[k])[1] for k in range(rank)]
        step = [1] * (rank - 1) + [per_unit]
        hlo = [[step[k] * int(rng.integers(0, min(3, sizes[k][c - 1] // step[k]) + 1)) if c > 0
                else step[k] * int(rng.integers(0, 3)) for c in range(ps[k])] for k in range(rank)]
        hhi = [[step[k] * int(rng.integers(0, min(3, sizes[k][c + 1] // step[k]) + 1)) if c + 1 < ps[k]
                else step[k] * int(rng.integers(0, 3)) for c in range(ps[k])] for k in range(rank)]
        opart = oracle.Partition(gs, ps, hlo, hhi)
        gpart = distdl.Partition(gs, ps, hlo, hhi, dtype=code)
    else:
        h = tuple(int(rng.integers(0, 3)) for _ in range(rank - 1)) + (per_unit * int(rng.integers(0, 2)),)
        opart = oracle.Partition(gs, ps, h, h, periodic)
        gpart = distdl.Partition(gs, ps, h, h, dtype=code, periodic=periodic)
    x32, y32 = random_shards(opart, 150 + seed), random_shards(opart, 180 + seed)
    if code == distdl.F32:
        x, y, add, back = x32, y32, None, host
        xs, ys = [dev(a) for a in x], [dev(a) for a in y]
    elif code == distdl.F64:
        x = [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in x32]
        y = [a.astype(np.float64) * (1.0 + 2.0 ** -33) for a in y32]
        xs, ys, add, back = [dev(a) for a in x], [dev(a) for a in y], None, host
    else:
        x = [inputs.f32_to_bf16_bits(a) for a in x32]
        y = [inputs.f32_to_bf16_bits(a) for a in y32]
        xs, ys, add, back = [_bits_dev(a) for a in x], [_bits_dev(a) for a in y], oracle.bf16_add, _bits_host
    distdl.halo_fwd(gpart, xs)
    distdl.halo_adj(gpart, ys)
    torch.cuda.synchronize()
    for a, b in zip(xs, oracle.halo_fwd_sequence(opart, x)):
        assert same_bits(back(a), b)
    for a, b in zip(ys, oracle.halo_adj_sequence(opart, y, add=add)):
        assert same_bits(back(a), b)


@pytest.mark.parametrize("seed", range(8))
def test_random_stencil_and_repartition_geometries(seed):
    rng = np.random.Generator(np.random.Philox(7100 + seed))
    R = int(rng.integers(1, 5))
    ps = tuple(int(rng.integers(1, 4)) for _ in range(3))
    gs = tuple(int(rng.integers(p * R, p * R + 40)) for p in ps)
    opart, obulk = oracle.Partition(gs, ps, R, R), oracle.Partition(gs, ps)
    gpart = distdl.Partition(gs, ps, (R,) * 3, (R,) * 3)
    w = inputs.normal((3, 2 * R + 1), 7200 + seed, 0.5)
    xg = inputs.normal(gs, 7300 + seed)
    x = oracle.scatter_global(opart, xg, fill=lambda wk: np.full(opart.padded_shape(wk), 1e30, dtype=np.float32))
    ys = [torch.empty(obulk.padded_shape(k), device=DEV) for k in range(opart.num_workers)]
    distdl.stencil3d_fwd(gpart, [dev(a) for a in x], w, ys)
    dy = oracle.scatter_global(obulk, inputs.normal(gs, 7400 + seed))
    dxs = [torch.full(opart.padded_shape(k), 5.0, device=DEV) for k in range(opart.num_workers)]
    distdl.stencil3d_adj(gpart, [dev(a) for a in dy], w, dxs)
    torch.cuda.synchronize()
    xz = oracle.scatter_global(opart, xg)
    eps = (6 * R + 5) * 2.0 ** -24
    for got, ref, mag in ((ys, oracle.stencil3d_fwd(opart, xz, w), oracle.stencil3d_fwd(opart, [np.abs(a) for a in xz], np.abs(w))),
                          (dxs, oracle.stencil3d_adj(opart, dy, w), oracle.stencil3d_adj(opart, [np.abs(a) for a in dy], np.abs(w)))):
        for a, b, m in zip(got, ref, mag):
            assert np.all(np.abs(host(a).astype(np.float64) - b) <= eps * m + 1e-30)
    # the same tensor from this partition to another random one and back
    ps2 = tuple(int(rng.integers(1, 4)) for _ in range(3))
    if all(g >= p for g, p in zip(gs, ps2)):
        rep = distdl.Repartition(gs, ps, ps2)
        odst = oracle.Partition(gs, ps2)
        src = oracle.scatter_global(obulk, xg)
        dst = [torch.empty(odst.padded_shape(k), device=DEV) for k in range(odst.num_workers)]
        back = [torch.empty(obulk.padded_shape(k), device=DEV) for k in range(obulk.num_workers)]
        distdl.repartition_fwd(rep, [dev(a) for a in src], dst)
        distdl.repartition_adj(rep, dst, back)
        torch.cuda.synchronize()
        for a, b in zip(dst, oracle.repartition_fwd(obulk, odst, src)):
            assert same_bits(host(a), b)
        for a, b in zip(back, src):
            assert same_bits(host(a), b)
