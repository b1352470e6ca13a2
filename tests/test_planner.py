"""Plans of the entry points without a GPU: the library's host code runs against stand-ins of the
CUDA calls (planner_probe.cpp, GB300's limits), and every call's plan is read back."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2505_22938_gb300", "csrc")
U8, U16, F32 = 0, 1, 2
IN, OUT = 1 << 32, 1 << 36  # addresses only: nothing is read or written


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("planner") / "planner_probe.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    cmd = ["g++", "-O1", "-std=c++17", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-x", "c++",
           os.path.join(HERE, "planner_probe.cpp"), "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda,
           "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    dll = ctypes.CDLL(so)
    dll.probe.restype = ctypes.c_longlong
    return dll


def disk(lib, r):
    k = ctypes.c_void_p()
    assert lib.fim_create_kernel_circle(r, ctypes.byref(k)) == 0
    return k


def ellipse(lib, a, b):
    k = ctypes.c_void_p()
    assert lib.fim_create_kernel_ellipse(a, b, ctypes.byref(k)) == 0
    return k


def plan(lib, *fields):
    return [lib.probe(f.encode()) for f in fields]


def outputs(n):
    return (ctypes.c_void_p * n)(*[OUT + (i << 32) for i in range(n)])


def percentiles(lib, k, dtype, w, h, pcts):
    v = (ctypes.c_double * len(pcts))(*pcts)
    return lib.fim_percentiles(ctypes.c_void_p(IN), outputs(len(pcts)), v, len(pcts), w, h,
                               ctypes.c_size_t(w << dtype), dtype, k, 0, None)


@pytest.mark.parametrize("dtype", [U8, U16, F32])
@pytest.mark.parametrize("size", [(256, 256), (1537, 1021), (4096, 4096)])
def test_quartiles_of_the_largest_disks_are_accepted(lib, dtype, size):
    """The tile of several target ranks holds all of them: a footprint beyond 65535 pixels stores
    ranks relative to the lowest target's, and the highest target's have to fit as well."""
    for r in range(96, 129):
        k = disk(lib, r)
        assert percentiles(lib, k, dtype, *size, (25.0, 50.0, 75.0)) == 0, r
        assert percentiles(lib, k, U16, *size, (5.0, 50.0, 95.0)) == 0 or r > 105, r
        lib.fim_destroy_kernel(k)


def radii(lib, dtype, w, h, rs):
    ks = [disk(lib, r) for r in rs]
    s = lib.fim_median_radii(ctypes.c_void_p(IN), outputs(len(rs)), (ctypes.c_void_p * len(rs))(*ks), len(rs), w, h,
                             ctypes.c_size_t(w << dtype), dtype, 0, None)
    for k in ks:
        lib.fim_destroy_kernel(k)
    return s


@pytest.mark.parametrize("dtype,rs", [(U16, range(65, 81)), (U8, range(65, 89)), (F32, range(65, 83))])
@pytest.mark.parametrize("size", [(1021, 763), (4096, 4096)])
def test_several_radii_keep_their_omnigram_in_shared_memory(lib, dtype, rs, size):
    """The disks' tables are part of the plan the tile is chosen by; float keys keep the 16-bit first pass
    (a plan that cannot sort by codes has no cheaper sort to fall back from)."""
    for r in rs:
        assert radii(lib, dtype, *size, (r // 2, r)) == 0
        assert plan(lib, "spilled", "codes") == [0, 0], r
        assert dtype != F32 or plan(lib, "sort") == [3], r


def test_several_radii_keep_their_resident_ctas(lib):
    """The words kept for the alignment of the disks' tables are given back before the launch."""
    assert radii(lib, U8, 3047, 5420, (15, 30)) == 0
    assert plan(lib, "threads", "resident") == [256, 4]


def median(lib, k, dtype, w, h):
    return lib.fim_median(ctypes.c_void_p(IN), ctypes.c_void_p(OUT), w, h, ctypes.c_size_t(w << dtype), dtype, k, 0,
                          None)


@pytest.mark.parametrize("dtype,r,size,tile", [
    (U8, 94, (587, 410), (64, 32)),       # all tiles at once: the height of least rows, not a taller one
    (F32, 117, (956, 539), (64, 64)),
    (U16, 43, (858, 447), (64, 56)),      # rows below the image count as well
    (U16, 128, (1537, 1021), (64, 64)),   # few waves of border tiles, omnigram in global scratch
    (U16, 97, (590, 1036), (64, 72)),
    (F32, 20, (2000, 1500), (32, 32)),    # less than three waves of the larger tiles
    (U16, 20, (2000, 1500), (32, 32)),
    (F32, 20, (4096, 4096), (64, 64)),
    (U16, 20, (4096, 4096), (32, 64)),
])
def test_tiles_of_images_of_few_waves(lib, dtype, r, size, tile):
    k = disk(lib, r)
    assert median(lib, k, dtype, *size) == 0
    assert tuple(plan(lib, "Tx", "Ty")) == tile
    lib.fim_destroy_kernel(k)


@pytest.mark.parametrize("size,sort,codes", [((448, 261), 3, 0), ((553, 296), 3, 0), ((3000, 2000), 2, 1)])
def test_float_images_of_border_tiles_keep_the_16_bit_pass(lib, size, sort, codes):
    k = disk(lib, 92)
    assert median(lib, k, F32, *size) == 0
    assert plan(lib, "sort", "codes", "spilled") == [sort, codes, 0]
    lib.fim_destroy_kernel(k)


def test_disk_of_256_box_rows_keeps_8_bit_coordinates(lib, monkeypatch):
    """r = 64 on 128 rows: the disk test's signed bytes do not reach every window centre."""
    monkeypatch.setenv("FIM_TILE", "64,128,8,2")
    k = disk(lib, 64)
    for dtype in (U8, U16, F32):
        assert median(lib, k, dtype, 2000, 1500) == 0
        assert plan(lib, "wide", "spilled") == [0, 0]
        assert radii(lib, dtype, 2000, 1500, (30, 64)) == 0
        assert plan(lib, "wide") == [1]
    lib.fim_destroy_kernel(k)


@pytest.mark.parametrize("dtype,r,tile", [
    (U8, 64, (64, 128)), (U16, 64, (64, 128)), (F32, 64, (64, 128)), (U16, 16, (32, 32)), (U16, 48, (64, 128)),
    (F32, 86, (64, 128)), (F32, 89, (64, 128)), (U8, 89, (64, 128)), (U8, 113, (64, 128)), (U16, 113, (64, 128)),
    (U16, 114, (64, 64)), (F32, 128, (64, 64))])
def test_tile_of_the_learned_bracket(lib, dtype, r, tile):
    """The tiles models have been trained on since the bracket exists: they do not follow the default
    shapes or the layout of a plan."""
    k = disk(lib, r)
    for size in ((300, 200), (4096, 4096)):
        assert lib.probe_bracket(k, dtype, *size) == 0
        assert tuple(plan(lib, "Tx", "Ty")) == tile
        assert plan(lib, "codes") == [0]
    lib.fim_destroy_kernel(k)


@pytest.mark.parametrize("dtype", [U8, U16, F32])
def test_ranks_of_the_learned_bracket(lib, dtype):
    """Its features are ranks over the footprint's size: whole up to 65535 pixels, 16 bits beyond."""
    for r in range(8, 129, 4):
        k = disk(lib, r)
        assert lib.probe_bracket(k, dtype, 4096, 4096) == 0
        n, base, top = plan(lib, "N", "rank_base", "rel_max")
        assert base == 0 if n <= 65535 else base > 0, r
        assert top >= min(n - 1, 65535), r
        lib.fim_destroy_kernel(k)


def noalloc(lib, k, dtype, w, h):
    return lib.fim_median_noalloc(ctypes.c_void_p(IN), ctypes.c_void_p(OUT), w, h, ctypes.c_size_t(w << dtype), dtype,
                                  k, 0, None)


def test_noalloc_keeps_its_tiles_and_its_calls(lib):
    """A float tile whose plan by codes does not fit the fixed workspace is planned without codes; spans
    kernels whose membership table leaves no room for a 512-thread tile take a 256-thread one."""
    for r in range(41, 61):
        k = disk(lib, r)
        assert noalloc(lib, k, F32, 4096, 4096) == 0
        assert plan(lib, "Tx", "Ty", "codes", "spilled") == [32, 64, 0, 0], r
        lib.fim_destroy_kernel(k)
    k = ellipse(lib, 104, 52)
    for dtype in (U8, U16, F32):
        for size in ((512, 512), (1537, 1021), (4096, 4096)):
            assert noalloc(lib, k, dtype, *size) == 0
    lib.fim_destroy_kernel(k)
    k = disk(lib, 100)
    assert noalloc(lib, k, F32, 4096, 4096) == 2  # beyond the workspace, as its test says
    lib.fim_destroy_kernel(k)


class Job(ctypes.Structure):
    _fields_ = [("src", ctypes.c_void_p), ("dst", ctypes.c_void_p), ("w", ctypes.c_int), ("h", ctypes.c_int),
                ("pitch", ctypes.c_size_t), ("dtype", ctypes.c_int), ("kernel", ctypes.c_void_p),
                ("percentile", ctypes.c_double)]


def batch(lib, dtype, rs):
    jobs = (Job * len(rs))()
    for i, r in enumerate(rs):
        jobs[i] = Job((1 << 40) + (i << 32), (1 << 42) + (i << 32), 1000, 900, 1000 << dtype, dtype, disk(lib, r).value,
                      -1.0)
    b = ctypes.c_void_p()
    lib.probe_forget_classes()
    assert lib.fim_batch_create(jobs, len(rs), ctypes.byref(b)) == 0


def test_batch_classes_keep_the_residency_of_their_tiles(lib):
    """The class kernels' static shared memory is part of a batch's plans, and a plan of fewer resident
    CTAs has a class of its own."""
    batch(lib, F32, [18, 30, 42, 45, 49])
    assert lib.probe_class(F32, 512, 5) == 2
    batch(lib, U16, [24, 28])
    assert lib.probe_class(U16, 512, 2) == 2
    batch(lib, U8, [36, 42, 53, 57, 95, 96])
    assert lib.probe_class(U8, 512, 4) == 2 and lib.probe_class(U8, 512, 2) == 1
    batch(lib, F32, [15, 16])
    assert lib.probe_class(F32, 256, 2) == 4
    batch(lib, U8, [2, 4, 8, 12, 16])  # six to eight CTAs: one class
    assert lib.probe_class(U8, 128, 5) >= 6


def test_plans_of_the_codes_tests_sort_by_codes(lib, monkeypatch):
    """Every plan of test_gpu_codes_interior.py, with at least two tiles whose box lies inside the image."""
    import numpy as np
    import test_gpu_codes_interior as t
    for dtype, spec, tile in t.PLANS:
        monkeypatch.setenv("FIM_TILE", tile)
        k = ctypes.c_void_p()
        if spec[0] == "polygon":
            xy = np.ascontiguousarray(spec[1], np.float64)
            assert lib.fim_create_kernel_polygon(xy.ctypes.data_as(ctypes.c_void_p), len(xy), ctypes.byref(k)) == 0
        else:
            k = disk(lib, spec[1]) if spec[0] == "circle" else ellipse(lib, *spec[1:])
        assert median(lib, k, {"u16": U16, "f32": F32}[dtype], t.W, t.H) == 0
        assert plan(lib, "codes") == [1], spec
        assert plan(lib, "inside")[0] >= 2, spec
        lib.fim_destroy_kernel(k)
