"""CPU tests of the host side of the library: the shared object loads and exports every symbol the
header declares, the planner's geometry and byte counts, and the error codes of the validation paths.
No kernel is launched here."""

import ctypes
import os
import re

import numpy as np
import pytest

import oracle
import paper_2006_03108_b200 as distdl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    names = set()
    inc = os.path.join(ROOT, "include")
    for header in sorted(os.listdir(inc)):
        if not header.endswith(".h"):
            continue
        text = open(os.path.join(inc, header)).read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        names.update(re.findall(r"\b(distdl_[a-z0-9_]+)\s*\(", text))
    return sorted(names)


def test_library_exports_every_declared_symbol():
    lib = ctypes.CDLL(distdl.LIB_PATH)
    names = _declared_symbols()
    assert len(names) >= 19
    for n in names:
        assert hasattr(lib, n), "libdistdl.so does not export %s" % n


APPENDIX_B = [
    # n, p, kernel, stride, pad -> halo_lo, halo_hi, unused_lo, unused_hi   (Figs. B1-B4)
    ((11, 3, 5, 1, 2), ([2, 2, 2], [2, 2, 2], [0, 0, 0], [0, 0, 0])),
    ((11, 3, 5, 1, 0), ([0, 1, 3], [3, 1, 0], [0, 0, 0], [0, 0, 0])),
    ((10, 3, 2, 2, 0), ([0, 0, 0], [0, 1, 0], [0, 0, 1], [0, 0, 0])),
    ((20, 6, 2, 2, 0), ([0] * 6, [0, 0, 1, 2, 1, 0], [0, 0, 0, 1, 2, 1], [0] * 6)),
]


@pytest.mark.parametrize("args,expect", APPENDIX_B)
def test_halo_widths_match_appendix_b_and_the_oracle(args, expect):
    n, p, k, s, pad = args
    got = distdl.halo_widths_1d(n, p, k, stride=s, pad_lo=pad, pad_hi=pad)
    assert tuple(got) == expect
    ref = oracle.halo_widths_1d(n, p, k, s, 1, pad, pad)
    assert list(got[0]) == [r["halo_lo"] for r in ref] and list(got[1]) == [r["halo_hi"] for r in ref]
    assert list(got[2]) == [r["unused_lo"] for r in ref] and list(got[3]) == [r["unused_hi"] for r in ref]


@pytest.mark.parametrize("n,p,k,s,d,pl,ph", [(37, 5, 3, 2, 2, 1, 0), (64, 7, 4, 3, 1, 2, 2), (9, 9, 3, 1, 1, 1, 1), (50, 4, 7, 1, 3, 0, 5)])
def test_halo_widths_random_cases_against_the_oracle(n, p, k, s, d, pl, ph):
    got = distdl.halo_widths_1d(n, p, k, stride=s, dilation=d, pad_lo=pl, pad_hi=ph)
    ref = oracle.halo_widths_1d(n, p, k, s, d, pl, ph)
    for i, key in enumerate(["halo_lo", "halo_hi", "unused_lo", "unused_hi"]):
        assert list(got[i]) == [r[key] for r in ref]


def test_shard_extents_match_the_oracle_partition():
    cases = [((11,), (3,), [2], [2]), ((67, 61, 68), (3, 2, 2), [2, 4, 4], [3, 4, 4]),
             ((9, 8), (2, 2), [[0, 4], [0, 3]], [[2, 0], [0, 0]])]
    for gs, ps, lo, hi in cases:
        g = distdl.Partition(gs, ps, lo, hi)
        o = oracle.Partition(gs, ps, lo, hi)
        assert g.num_workers == o.num_workers
        for w in range(o.num_workers):
            st, bulk, padded, hl, hh = g.shard_extents(w)
            assert st == o.bulk_start(w) and bulk == o.bulk_shape(w) and padded == o.padded_shape(w)
            assert (hl, hh) == o.widths(w)


def test_plan_bytes_of_the_baseline_configurations():
    # 2-D: 4 shards of 130^2, width 1.  3-D: 64 shards of 136^3, width 4.
    p1 = distdl.Partition((256, 256), (2, 2), (1, 1), (1, 1))
    assert p1.halo_stats(False) == (32, 32, 12368)
    assert p1.halo_stats(True)[2] == 20528
    p3 = distdl.Partition((512,) * 3, (4,) * 3, (4,) * 3, (4,) * 3)
    boxes, tiles, nbytes = p3.halo_stats(False)
    assert boxes == 64 * 26 and nbytes == 186177536
    assert p3.halo_stats(True)[2] == 330205184
    # independent count: ghost cells written + interior ghost cells read (fp32)
    ghost = 64 * (136 ** 3 - 128 ** 3)
    interior = sum(np.prod([min(s + 132, 512) - max(s - 4, 0) for s in (a, b, c)]) - 128 ** 3
                   for a in range(0, 512, 128) for b in range(0, 512, 128) for c in range(0, 512, 128))
    assert nbytes == 4 * (ghost + int(interior))


def _status(fn, *a, **k):
    with pytest.raises(distdl.DistdlError) as e:
        fn(*a, **k)
    return e.value.status


def test_partition_validation_errors():
    assert _status(distdl.Partition, (4, 4), (8, 1)) == 2                       # fewer cells than workers
    assert _status(distdl.Partition, (8, 8), (4, 1), (3, 0), (0, 0)) == 2        # ghost wider than the neighbour
    assert _status(distdl.Partition, (8,) * 6, (1,) * 6) == 1                    # rank > 5
    assert _status(distdl.Partition, (1024, 1024), (32, 32)) == 4                # > 256 workers
    assert _status(distdl.Partition, (8, 8), (2, 2), (-1, 0), (0, 0)) == 2
    assert _status(distdl.halo_widths_1d, 4, 2, 9) == 2                          # kernel larger than the input


class _FakeTensor:
    """Stands in for a device tensor: only the address and the size are looked at before launch."""

    def __init__(self, addr, numel=16):
        self._addr, self._n = addr, numel
        import torch
        self.dtype = torch.float32

    def data_ptr(self):
        return self._addr

    def numel(self):
        return self._n


def test_operator_argument_validation_without_a_device():
    ok, odd = _FakeTensor(0x10000), _FakeTensor(0x10004)
    assert _status(distdl.broadcast_fwd, odd, [ok], stream=0) == 3               # alignment
    assert _status(distdl.broadcast_fwd, ok, [odd], stream=0) == 3
    assert _status(distdl.sumreduce_fwd, [ok, _FakeTensor(0)], ok, stream=0) == 1  # NULL source
    assert _status(distdl.sumreduce_fwd, [_FakeTensor(0x20000), ok], ok, stream=0) == 1  # dst aliases source 1
    part = distdl.Partition((8, 8), (2, 2), (1, 1), (1, 1))
    import torch
    if not torch.cuda.is_available():
        # created without a device: geometry works, operators refuse
        assert _status(distdl.halo_fwd, part, [ok] * 4, stream=0) == 5
    lib = distdl.lib()
    vp = ctypes.c_void_p
    arr = (vp * 4)(0x10000, 0x20000, 0x30000, 0x40000)
    assert lib.distdl_affine_fwd(16, 100, 128, 1, 1, arr, arr, None, arr, None) == 4   # block not a multiple of 8
    assert lib.distdl_affine_fwd(16, 256, 256, 3, 1, arr, arr, None, arr, None) == 2   # not divisible by the grid
    assert lib.distdl_conv_fwd(part.handle, arr, vp(0x50000), None, 3, 3, arr, None) == 2  # not a rank-4 partition
    p4 = distdl.Partition((1, 2, 16, 16), (1, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))
    assert lib.distdl_conv_fwd(p4.handle, arr, vp(0x50000), None, 3, 3, arr, None) == 2    # widths do not match 3x3
    assert lib.distdl_conv_fwd(p4.handle, arr, vp(0x50000), None, 4, 4, arr, None) == 4    # even kernel
    assert lib.distdl_last_error().decode() != ""


def test_validation_of_the_gradient_stencil_and_dtype_entry_points():
    lib = distdl.lib()
    vp = ctypes.c_void_p
    arr = (vp * 16)(*[0x10000 * (i + 1) for i in range(16)])
    # affine parameter gradients
    assert lib.distdl_affine_adj_params(16, 100, 128, 1, 1, arr, arr, arr, None, None) == 4   # block not a multiple of 8
    assert lib.distdl_affine_adj_params(16, 256, 256, 3, 1, arr, arr, arr, None, None) == 2   # not divisible by the grid
    assert lib.distdl_affine_adj_params(16, 256, 256, 1, 1, None, arr, arr, None, None) == 1  # NULL argument
    odd = (vp * 1)(0x10004)
    assert lib.distdl_affine_adj_params(16, 128, 128, 1, 1, odd, arr, arr, None, None) == 3   # alignment
    # convolution parameter gradients: the geometry is checked before anything touches a device
    p2 = distdl.Partition((8, 8), (2, 2), (1, 1), (1, 1))
    p4 = distdl.Partition((1, 2, 16, 16), (1, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))
    n = ctypes.c_int64(0)
    assert lib.distdl_conv_adj_params_workspace(p2.handle, 3, 3, ctypes.byref(n)) == 2          # not rank 4
    assert lib.distdl_conv_adj_params_workspace(p4.handle, 3, 3, ctypes.byref(n)) == 2          # widths do not match 3x3
    assert lib.distdl_conv_adj_params_workspace(p4.handle, 4, 4, ctypes.byref(n)) == 4          # even kernel
    assert lib.distdl_conv_adj_params_workspace(p4.handle, 5, 5, None) == 1
    assert lib.distdl_conv_adj_params(p4.handle, arr, arr, 5, 5, vp(0x50000), None, None, 0, None) == 1   # no workspace
    # star stencil
    taps = (ctypes.c_float * 27)(*([0.5] * 27))
    p3 = distdl.Partition((8, 8, 8), (2, 1, 1), (2, 2, 2), (2, 2, 2))
    assert lib.distdl_stencil3d_fwd(p2.handle, arr, taps, 1, arr, None) == 2                    # not rank 3
    assert lib.distdl_stencil3d_fwd(p3.handle, arr, taps, 5, arr, None) == 4                    # radius beyond 4
    assert lib.distdl_stencil3d_fwd(p3.handle, arr, taps, 1, arr, None) == 2                    # halo width is not the radius
    assert lib.distdl_stencil3d_adj(p3.handle, arr, None, 2, arr, None) == 1
    odd8 = (vp * 2)(0x10008, 0x20000)
    assert lib.distdl_stencil3d_fwd(p3.handle, odd8, taps, 2, arr, None) == 3                   # alignment
    with pytest.raises(ValueError):
        distdl.stencil3d_fwd(p3, [], [[1.0, 2.0]] * 3, [])                                      # even tap count
    # element types
    assert lib.distdl_sumreduce_fwd(arr, vp(0x90000), 2, 8, 7, None) == 1                       # unknown dtype
    assert lib.distdl_broadcast_fwd(vp(0x90000), arr, 2, 8, 7, None) == 1
    p64 = distdl.Partition((9, 9), (2, 2), (1, 1), (1, 1), dtype=distdl.F64)
    assert p64.halo_stats(False)[2] == 2 * distdl.Partition((9, 9), (2, 2), (1, 1), (1, 1)).halo_stats(False)[2]
    r64 = distdl.Repartition((12, 8), (3, 1), (1, 2), distdl.F64)
    assert r64.shard_shape(0) == (4, 8) and r64.shard_shape(1, destination=True) == (12, 4)


def test_periodic_partition_geometry_and_refusals():
    lib = distdl.lib()
    vp = ctypes.c_void_p
    # 8 x 8 on 2 x 2 workers, width 1: 20 ghost cells per shard; all of them have an owner when both
    # dimensions wrap (20 reads + 20 writes of 4 bytes per shard), only 9 of them (a row, a column, a corner) otherwise
    per = distdl.Partition((8, 8), (2, 2), (1, 1), (1, 1), periodic=(True, True))
    flat = distdl.Partition((8, 8), (2, 2), (1, 1), (1, 1))
    assert per.halo_stats(False)[2] == 4 * (20 + 20) * 4
    assert flat.halo_stats(False)[2] == 4 * (20 + 9) * 4
    # adjoint: every ghost read and cleared (8 B), every bulk cell in reach of a face read and written (8 B):
    # all 12 cells of the bulk's rim with both dimensions periodic, 7 of them (one row, one column) otherwise
    assert per.halo_stats(True)[2] == 4 * (20 * 8 + 12 * 8)
    assert flat.halo_stats(True)[2] == 4 * (20 * 4 + 9 * 4 + 7 * 8)
    # the ghost-width rule holds across the seam as well
    assert _status(distdl.Partition, (6,), (2,), (4,), (0,), periodic=(True,)) == 2
    # a worker alone along a periodic dimension is its own neighbour
    one = distdl.Partition((7,), (1,), (2,), (3,), periodic=(True,))
    assert one.halo_stats(False)[2] == (5 + 5) * 4 and one.halo_stats(True)[0] >= 1
    # fused layers take no periodic partitions
    arr = (vp * 16)(*[0x10000 * (i + 1) for i in range(16)])
    p4 = distdl.Partition((1, 2, 16, 16), (1, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2), periodic=(False, False, True, True))
    assert lib.distdl_conv_fwd(p4.handle, arr, vp(0x50000), None, 5, 5, arr, None) == 4
    p3 = distdl.Partition((8, 8, 8), (2, 1, 1), (2, 2, 2), (2, 2, 2), periodic=(True, False, False))
    taps = (ctypes.c_float * 15)(*([0.5] * 15))
    assert lib.distdl_stencil3d_fwd(p3.handle, arr, taps, 2, arr, None) == 4


def test_validation_of_the_generalized_convolution():
    lib = distdl.lib()
    vp = ctypes.c_void_p
    arr = (vp * 64)(*[0x10000 * (i + 1) for i in range(64)])
    px = distdl.Partition((1, 4, 16, 16), (1, 2, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))
    assert lib.distdl_convg_fwd(px.handle, 6, 2, arr, arr, None, 3, 3, arr, None) == 2          # widths do not match 3x3
    assert lib.distdl_convg_fwd(px.handle, 6, 2, arr, arr, None, 4, 4, arr, None) == 4          # even kernel
    assert lib.distdl_convg_fwd(px.handle, 1, 2, arr, arr, None, 5, 5, arr, None) == 2          # fewer channels than blocks
    assert lib.distdl_convg_fwd(px.handle, 18, 9, arr, arr, None, 5, 5, arr, None) == 4         # more than 8 channel blocks
    assert lib.distdl_convg_adj(px.handle, 6, 2, None, arr, 5, 5, arr, None) == 1
    pb = distdl.Partition((2, 4, 16, 16), (2, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))
    assert lib.distdl_convg_fwd(pb.handle, 6, 2, arr, arr, None, 5, 5, arr, None) == 4          # batch partitioned
    odd = (vp * 8)(*[0x10004 + 0x10000 * i for i in range(8)])
    assert lib.distdl_convg_fwd(px.handle, 6, 2, odd, arr, None, 5, 5, arr, None) == 3          # alignment


def test_header_compiles_as_c_and_the_library_links_from_c(tmp_path):
    import shutil
    import subprocess
    gcc = shutil.which("gcc")
    if gcc is None:
        pytest.skip("no C compiler")
    exe = str(tmp_path / "host_check")
    libdir = os.path.dirname(distdl.LIB_PATH)
    subprocess.check_call([gcc, "-std=c99", "-Wall", "-Werror", "-I", os.path.join(ROOT, "include"),
                           os.path.join(ROOT, "tests", "c_abi", "host_check.c"), "-o", exe,
                           "-L", libdir, "-ldistdl", "-Wl,-rpath," + libdir])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout + out.stderr


@pytest.mark.parametrize("gs,ps,lo,hi", [
    ((512, 512, 512), (4, 4, 4), (4, 4, 4), (4, 4, 4)),
    ((256, 256), (2, 2), (1, 1), (1, 1)),
    ((70, 66, 72), (2, 3, 2), (4, 2, 3), (1, 4, 2)),
    ((37, 45), (3, 2), (2, 1), (1, 3)),
    ((9, 40), (4, 1), (2, 3), (2, 0)),            # shards as thin as their neighbours' ghosts
    ((16, 16, 1024, 1024), (1, 1, 4, 4), (0, 0, 2, 2), (0, 0, 2, 2)),
])
def test_bench_byte_counts_from_oracle_geometry_match_the_planner(gs, ps, lo, hi):
    """bench.py counts the algorithmic bytes of H, H* and the convolution from partition geometry alone (the
    oracle's Partition, or its own extents-only stand-in); the library's planner counts them from its box lists."""
    import bench
    gp = distdl.Partition(gs, ps, lo, hi)
    want = (gp.halo_stats(False)[2], gp.halo_stats(True)[2])
    assert bench.halo_algorithmic_bytes(oracle.Partition(gs, ps, lo, hi)) == want
    assert bench.halo_algorithmic_bytes(bench._Geometry(gs, ps, lo, hi)) == want
    if len(gs) == 4:
        a = bench.conv_algorithmic_bytes(oracle.Partition(gs, ps, lo, hi))
        assert a == bench.conv_algorithmic_bytes(bench._Geometry(gs, ps, lo, hi)) == 2172796928


def test_bench_reference_arm_does_not_load_the_cuda_library():
    """`bench.py --impl reference` and the CPU-baseline leg time the oracle alone."""
    import subprocess, sys
    code = ("import sys, bench; b, s, per = bench.oracle_sample_step(bench.ORACLE_LEVELS[2]); "
            "import paper_2006_03108_b200 as d; assert d._lib is None, 'library was loaded'; "
            "assert b > 0 and s > 0; print('ok')")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr


def test_partition_broadcast_rejects_shapes_that_do_not_broadcast():
    lib = distdl.lib()
    one = ctypes.c_void_p(256)
    ptrs = (ctypes.c_void_p * 8)(*[256] * 8)
    elems = (ctypes.c_int64 * 8)(*[4] * 8)

    def call(src_p, dst_p):
        r = len(src_p)
        return lib.distdl_partition_broadcast_fwd(r, (ctypes.c_int32 * r)(*src_p), (ctypes.c_int32 * r)(*dst_p), elems,
                                                  ptrs, ptrs, distdl.F32, None)
    assert call((2, 2), (4, 2)) == 2 and b"dimension 0" in lib.distdl_last_error()       # DISTDL_ERR_SHAPE
    assert call((2, 1), (1, 2)) == 2
    assert call((1,), (512,)) == 4                                                        # DISTDL_ERR_UNSUPPORTED
    assert lib.distdl_partition_broadcast_fwd(1, None, None, elems, ptrs, ptrs, distdl.F32, None) == 1


@pytest.mark.parametrize("gradients", [False, True])
@pytest.mark.parametrize("k", [3, 5, 7])
def test_depthwise_convolution_copies_end_inside_their_arrays(k, gradients):
    """Rows of arrays without ghosts travel in 16-byte blocks: none may begin before the array's end and reach past it.  The rows whose
    last block would are the few of the last 12 bytes; they travel in their whole blocks and single cells."""
    h = (0, 0, k // 2, k // 2)
    for planes in (1, 2, 3, 4):
        for rows in range(1, 12):
            for cols in (1, 2, 3, 4, 5, 9, 66, 130):
                part = distdl.Partition((1, planes, rows, cols), (1, 1, 1, 1), h, h)
                past, by_cell = distdl.selftest_conv_row_reads(part, k, gradients)
                assert past <= 0 and by_cell <= 3, (planes, rows, cols, past, by_cell)
    if k == 3:
        part = distdl.Partition((1, 1, 6, 3), (1, 1, 1, 3), h, h)
        past, by_cell = distdl.selftest_conv_row_reads(part, k, gradients)
        assert past <= 0 and by_cell <= 3 * 3
    for parts in ((1, 1), (2, 3)):
        for cols in range(3 * parts[1], 280):                    # the last row ends anywhere in a block, in strips of 64 and 128 columns
            part = distdl.Partition((1, 701 if cols > 200 else 1, 3 * parts[0], cols), (1, 1) + parts, h, h)
            past, cut = distdl.selftest_conv_row_reads(part, k, gradients)
            assert past <= 0 and (cut > 0 or cols % 4 == 0 or parts != (1, 1)), (parts, cols, past, cut)


def test_every_kernel_waits_for_the_stream_before_it_touches_memory():
    """Kernels are launched while their predecessors in the stream run; what those wrote is visible to a kernel only after its
    own wait.  So every kernel launched that way begins with stream_enter(), under no condition, and nothing else lets
    successors in.  A few set themselves up ahead of it, with nothing but their launch's parameters, shared and tensor memory."""
    src = os.path.join(ROOT, "paper_2006_03108_b200", "csrc")
    bodies, triggers = {}, 0
    for name in sorted(os.listdir(src)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(src, name)).read())
        triggers += text.count("griddepcontrol.launch_dependents")
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", text):
            brace = text.index("{", m.end())
            depth, end = 1, brace + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            bodies[m.group(1)] = text[brace + 1:end - 1]
    bodies.pop("selftest_wait_kernel")          # launched the ordinary way
    assert triggers == 1 and len(bodies) >= 20 and "halo_adj_kernel" in bodies
    for kernel, body in sorted(bodies.items()):
        assert len(re.findall(r"^    stream_enter\(\);", body, re.M)) == 1, kernel
        assert body.count("stream_enter") == 1 and body.count("griddepcontrol") == 0, kernel
        before = re.sub(r"static_assert\([^;]*;|constexpr [^;]*;|extern __shared__ [^;]*;", "", body[:body.index("stream_enter();")])
        if kernel not in ("convg_kernel", "affine_kernel_pair", "affine_kernel_split", "affine_kernel_quad", "affine_dw_kernel"):
            assert not before.strip(), kernel
            continue
        assert not re.search(r"__ldg|cp_async|bulk|tma_|atomic|\bld_|\bst_|\breturn\b", before), kernel
        assert not re.search(r"\b[GPQ]\.(p\.)?(in|out|w|x|y|dx|dy|dw|db|bias|partial|\w*map)\b", before), kernel      # what points to device memory
        assert all(re.match(r"tcgen05\.(alloc|relinquish_alloc_permit)\.", a) for a in re.findall(r'asm volatile\("([^"]*)"', before)), kernel
        assert set(re.findall(r"\b(\w+)\[[^\]]*\] = ", before)) <= {"table", "tiles", "wbuf"}, kernel
        assert set(re.findall(r"\*(\w+) = ", before)) - {"aligned", "bars", "tmem_slot", "abort_flag", "tiles", "wbuf", "table", "ptrs"} == set(), kernel


def test_calls_check_their_arguments_before_the_library_sees_them():
    """Lists that are too short are errors, not whatever lies behind them; wrong types are exceptions."""
    part = distdl.Partition((8, 8), (2, 2), (1, 1), (1, 1))
    y, few = [256] * 4, [256, 512]
    conv = distdl.Partition((1, 1, 8, 8), (1, 1, 2, 2), (0, 0, 1, 1), (0, 0, 1, 1))
    w = np.zeros((1, 3, 3))
    w_ptr = type("W", (), {"shape": w.shape, "data_ptr": lambda self: 1024})()
    for shards in (few, tuple(few), [None] * 4, []):
        with pytest.raises(distdl.DistdlError) as e:
            distdl.conv_fwd(conv, shards, w_ptr, None, y, stream=0)
        assert e.value.status == 1
    with pytest.raises(AttributeError):
        distdl.halo_fwd(part, ["shard"] * 4, stream=0)
    with pytest.raises(TypeError):
        distdl.pool_fwd(conv, y, (3.5, 3), (1, 1), ((1, 1), (1, 1)), distdl.POOL_MAX, y, stream=0)
    with pytest.raises(ValueError):
        distdl.stencil3d_fwd(part, y, [[1, 2, 3], [1, 2, 3], [1, 2]], y, stream=0)
    conv.close()
    conv.close()
    for call in (lambda: distdl.conv_fwd(conv, y, w_ptr, None, y, stream=0), lambda: distdl.halo_adj(conv, y, stream=0)):
        with pytest.raises(distdl.DistdlError) as e:
            call()
        assert e.value.status == 1
    raw, radius = distdl._taps(np.arange(9).reshape(3, 3))
    assert radius == 1 and np.array_equal(np.frombuffer(raw, np.float32), np.arange(9, dtype=np.float32))


def _fused_pool_adjoint_disagreements(kernel, stride, dim, sizes, paddings):
    """Layers in which a row (dim 0) or column (dim 1) of some worker's bulk gets other outputs than those whose windows hold it, and the
    number of layers of which that was asked."""
    wrong, asked = [], 0
    for n in sizes:
        for p in range(1, 9):
            for pad in paddings:
                m = (n + sum(pad) - kernel) // stride + 1
                if n < p or m < p:
                    continue
                lo, hi = distdl.halo_widths_1d(n, p, kernel, stride, pad_lo=pad[0], pad_hi=pad[1])[:2]
                across = distdl.halo_widths_1d(16, 1, kernel, stride, pad_lo=pad[0], pad_hi=pad[1])[:2]
                shape, parts, los, his = [1, 1, 16, 16], [1] * 4, [0, 0, across[0], across[0]], [0, 0, across[1], across[1]]
                shape[2 + dim], parts[2 + dim], los[2 + dim], his[2 + dim] = n, p, lo, hi
                try:
                    part = distdl.Partition(shape, parts, los, his)
                except distdl.DistdlError:
                    continue                                     # ghosts wider than a neighbour
                for w in range(p):
                    fused, got = distdl.selftest_pool_adj_terms(part, kernel, stride, pad, distdl.POOL_AVG, w, dim)
                    if not fused:
                        break
                    start, size = (v[2 + dim] for v in part.shard_extents(w)[:2])
                    at = start + pad[0] + np.arange(size)[:, None] - np.arange(kernel)[None, :]       # first cell of the window, padded
                    want = np.where((at >= 0) & (at % stride == 0) & (at // stride < m), at // stride, -1)
                    if not np.array_equal(np.array(got), want):
                        wrong.append((n, p, pad, w))
                        break
                else:
                    asked += 1
    return wrong, asked


@pytest.mark.parametrize("dim", [0, 1])
@pytest.mark.parametrize("kernel,stride", [(2, 2), (3, 2), (3, 1)])
def test_fused_pool_adjoint_adds_every_output_that_holds_a_cell(kernel, stride, dim):
    """Windows meet shard ends in as many ways as there are widths, partitions and paddings: all of them up to 160, and further on around
    the widths whose shards end a strip of 64 or 128 columns or begin the next.  A shard that begins with a whole window of the worker on its
    left (2 x 2 / 2, 20 columns on 4 workers) once got no gradient in its first two columns; one of 128 m + 1 columns (3 x 3 / 2, 257 on 2 workers, padded on
    the left) lost a term of the column before its last."""
    paddings = [(a, b) for a in range(kernel) for b in range(kernel)]
    wrong, asked = _fused_pool_adjoint_disagreements(kernel, stride, dim, range(kernel, 161), paddings)
    ends = sorted({p * at + d for p in range(1, 9) for at in (64, 128) for d in range(-4, 5) if p * at + d > 160})
    more = _fused_pool_adjoint_disagreements(kernel, stride, dim, ends + [1020, 1021, 1022, 1023, 1024], paddings)
    assert not wrong + more[0], (len(wrong + more[0]), wrong[:3], more[0][:3])
    assert asked > 1000 and more[1] > 1000


@pytest.mark.parametrize("kernel,stride,mode,shape,parts,fused", [
    # B200, adjoint, one kernel against two (us)
    (2, 2, "avg", (512, 16, 14, 14), (1, 2), False),             # 59.6 / 27.5
    (2, 2, "max", (64, 16, 62, 62), (2, 2), False),              # 25.2 / 17.6
    (3, 2, "max", (256, 16, 62, 62), (2, 2), False),             # 105 / 77
    (3, 1, "avg", (256, 16, 30, 30), (2, 2), False),             # 91.7 / 86.9
    (2, 2, "avg", (4, 16, 258, 258), (4, 4), True),              # 10.5 / 12.1
    (2, 2, "max", (12, 16, 362, 358), (2, 3), True),             # 36.1 / 39.5
    (3, 2, "max", (16, 16, 1024, 1024), (4, 4), True),           # 350 / 417
    (3, 2, "avg", (128, 16, 126, 126), (2, 2), True),            # 68.7 / 77.8
    (3, 1, "max", (32, 16, 126, 126), (2, 2), True),             # 40.9 / 75.3
])
def test_pool_adjoint_takes_the_faster_of_one_kernel_and_two(kernel, stride, mode, shape, parts, fused):
    pad = (0, 0) if kernel == 2 else (1, 1)
    w = [distdl.halo_widths_1d(shape[2 + d], parts[d], kernel, stride, pad_lo=pad[0], pad_hi=pad[1]) for d in range(2)]
    part = distdl.Partition(shape, (1, 1) + parts, [0, 0, w[0][0], w[1][0]], [0, 0, w[0][1], w[1][1]])
    code = distdl.POOL_AVG if mode == "avg" else distdl.POOL_MAX
    assert distdl.selftest_pool_adj_terms(part, kernel, stride, pad, code, 0, 0)[0] == (2 if fused else 1)


class _Change:
    """A number whose conversion changes the list that it is in."""

    def __init__(self, change):
        self.change = change

    def __float__(self):
        self.change()
        return 2.0


def test_taps_that_change_while_they_are_read():
    for at in range(3):
        rows = [[1.0] * 5 for _ in range(3)]
        rows[at][1] = _Change(rows[at].clear)
        with pytest.raises(ValueError):
            distdl._taps(rows)
        rows = [[1.0] * 5 for _ in range(3)]
        rows[at][4] = _Change(rows.clear)
        if at < 2:
            with pytest.raises(ValueError):
                distdl._taps(rows)
        else:
            assert np.array_equal(np.frombuffer(distdl._taps(rows)[0], np.float32), [1] * 14 + [2])


class _Block:
    """A block of weights at some address."""

    def __init__(self, *shape):
        self.shape = shape

    def data_ptr(self):
        return 0x10000

    def numel(self):
        return 1 << 20

    def element_size(self):
        return 1


def test_short_lists_are_refused_whatever_they_hold():
    """Also where an entry may be missing (bias, positions, db), and where the list is as long as the calls' own array."""
    a, w = [0x10000 * (i + 1) for i in range(256)], _Block(3, 3, 5, 5)

    def refuses(needed, fn, *args):
        with pytest.raises(distdl.DistdlError, match="%d are needed" % needed) as e:
            fn(*args, stream=0)
        assert e.value.status == 1

    for workers in (65, 100, 256):
        part = distdl.Partition((1024,), (workers,), (1,), (1,))
        for n in {0, 10, 63, 64, workers - 1}:
            refuses(workers, distdl.halo_fwd, part, a[:n])
            refuses(workers, distdl.halo_adj, part, tuple(a[:n]))
    rep = distdl.Repartition((8, 8), (4, 1), (1, 2))
    refuses(4, distdl.repartition_fwd, rep, a[:3], a[:2])
    refuses(2, distdl.repartition_fwd, rep, a[:4], a[:1])
    refuses(2, distdl.repartition_adj, rep, a[:1], a[:4])
    conv = distdl.Partition((1, 1, 8, 8), (1, 1, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))
    refuses(4, distdl.conv_fwd, conv, a[:4], w, None, a[:3])
    refuses(4, distdl.conv_adj, conv, a[:3], w, a[:4])
    refuses(4, distdl.conv_adj_params, conv, a[:4], a[:2], (5, 5), 256, None, w)
    px = distdl.Partition((1, 6, 16, 16), (1, 2, 2, 2), (0, 0, 2, 2), (0, 0, 2, 2))            # 8 input shards, 12 output shards, 6 blocks
    for lists, needed in [((a[:7], [w] * 6, a[:3], a[:12]), 8), ((a[:8], [w] * 5, None, a[:12]), 6), ((a[:8], [w] * 6, [None] * 2, a[:12]), 3),
                          ((a[:8], [w] * 6, None, a[:11]), 12)]:
        refuses(needed, distdl.convg_fwd, px, 9, 3, *lists)
    refuses(12, distdl.convg_adj, px, 9, 3, a[:11], [w] * 6, a[:8])
    refuses(8, distdl.convg_adj, px, 9, 3, a[:12], [w] * 6, a[:7])
    refuses(3, distdl.convg_adj_params, px, 9, 3, a[:8], a[:12], (5, 5), a[:6], a[:2], w)
    refuses(6, distdl.convg_adj_params, px, 9, 3, a[:8], a[:12], (5, 5), a[:5], None, w)
    st = distdl.Partition((8, 8, 8), (2, 1, 1), (1, 1, 1), (1, 1, 1))
    refuses(2, distdl.stencil3d_fwd, st, a[:2], np.ones((3, 3)), a[:1])
    refuses(2, distdl.stencil3d_adj, st, a[:1], np.ones((3, 3)), a[:2])
    pool = distdl.Partition((1, 1, 8, 8), (1, 1, 2, 2))
    layer = ((2, 2), (2, 2), ((0, 0), (0, 0)))
    refuses(4, distdl.pool_fwd, pool, a[:4], *layer, distdl.POOL_MAX, a[:4], a[:3])
    refuses(4, distdl.pool_adj, pool, a[:4], a[:3], *layer, distdl.POOL_MAX, a[:4])
    refuses(4, distdl.pool_fwd, pool, a[:4], *layer, distdl.POOL_AVG, a[:3])
    refuses(2, distdl.affine_fwd, 16, 256, 256, 2, 4, a[:4], a[:8], [None], a[:2])
    refuses(4, distdl.affine_fwd, 16, 256, 256, 2, 4, a[:3], a[:8], None, a[:2])
    refuses(8, distdl.affine_adj, 16, 256, 256, 2, 4, a[:2], a[:7], a[:4])
    refuses(2, distdl.affine_adj_params, 16, 256, 256, 2, 4, a[:2], a[:4], a[:8], a[:1])
    t = [_FakeTensor(v) for v in a]
    refuses(4, distdl.partition_broadcast_fwd, (2, 1), (2, 2), t[:2], t[:3])
    refuses(2, distdl.partition_broadcast_fwd, (2, 1), (2, 2), t[:1], t[:4])
    refuses(4, distdl.partition_broadcast_adj, (2, 1), (2, 2), t[:3], t[:2])
    with pytest.raises(distdl.DistdlError, match="4 are needed"):
        distdl.halo_fwd_noalloc((8, 8), (2, 2), (1, 1), (1, 1), t[:3], stream=0)


def test_extension_is_named_after_the_interpreter_it_is_built_for():
    import sysconfig
    assert os.path.basename(distdl._load().__file__) == "_binding" + sysconfig.get_config_var("EXT_SUFFIX")


def test_prototypes_agree_with_the_headers():
    """distdl.lib() gives the library's functions to callers of their own; csrc/binding.cpp takes the types from the headers themselves."""
    text = "".join(open(os.path.join(ROOT, "include", h)).read() for h in ("distdl.h", "distdl_selftest.h"))
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    scalars = {"int32_t": ctypes.c_int32, "int64_t": ctypes.c_int64, "distdl_dtype_t": ctypes.c_int32, "size_t": ctypes.c_size_t}
    kinds = {ctypes.POINTER(ctypes.c_int32): "int32_t*", ctypes.POINTER(ctypes.c_int64): "int64_t*", ctypes.POINTER(ctypes.c_float): "float*",
             ctypes.POINTER(ctypes.POINTER(ctypes.c_int32)): "int32_t**"}
    seen = set()
    for name, args in re.findall(r"\b(distdl_[a-z0-9_]+)\s*\(([^()]*)\)\s*;", text):
        types = getattr(distdl.lib(), name).argtypes
        if types is None:
            continue
        seen.add(name)
        declared = [] if args.strip() in ("", "void") else [re.sub(r"\bconst\b|\s", "", re.sub(r"\w+\s*$", "", a.strip())) for a in args.split(",")]
        assert len(declared) == len(types), name
        for want, got in zip(declared, types):
            if want in scalars:
                assert got is scalars[want], (name, want)
            elif want.rstrip("*") in ("int32_t", "int64_t", "float"):
                assert kinds[got] == want, (name, want)
            else:                                            # handles, buffers: void *; arrays of them: void **
                assert got is (ctypes.POINTER(ctypes.c_void_p) if want.endswith("**") else ctypes.c_void_p), (name, want)
    assert len(seen) >= 40, sorted(seen)
