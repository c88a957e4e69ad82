"""The library's host code without a GPU: which kernels a call launches, what
it allocates and keeps, and what it does when the runtime refuses a request.
Each test runs in a process of its own on a stand-in for the CUDA runtime
(fake_cudart.c), which notes the calls and runs no kernel."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2110_12952_gb300 import build, capi, workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))

pytestmark = pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "bin", "nvcc")) or shutil.which("gcc") is None,
                                reason="nvcc or gcc not available")

PRELUDE = """
import ctypes, re
from ctypes import byref, c_int, c_int32, c_int64, c_void_p
fake = ctypes.CDLL({fake!r}, mode=ctypes.RTLD_GLOBAL)
lib = ctypes.CDLL({lib!r})
fake.fake_log.restype, lib.fractal_last_error.restype = ctypes.c_char_p, ctypes.c_char_p
fake.fake_held.restype, fake.fake_limit.argtypes = ctypes.c_size_t, [ctypes.c_size_t]
TABLES = {tables!r}
A, B = 1 << 40, 1 << 41          # where a program's buffers might be: no kernel runs

def handle(name, r):
    k, s, dim, table = TABLES[name]
    h = c_void_p()
    assert lib.fractal_create(k, s, r, dim, (c_int32 * len(table))(*table), byref(h)) == 0, lib.fractal_last_error()
    return h

def step(h, steps, stream=0, rule=(8, 12), src=A, dst=B, fn="fractal_step"):
    return getattr(lib, fn)(h, c_void_p(src), c_void_p(dst), c_int64(steps), *rule, c_void_p(stream))

def log(pattern="", clear=True):
    lines = [x for x in fake.fake_log().decode().split("\\n") if re.search(pattern, x)]
    if clear:
        fake.fake_clear()
    return [x for x in lines if x]

def kernels():
    return [x.split()[1] for x in log("^launch")]

def sliced(names):
    return any("slice_" in x for x in names)
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("fake_cudart")
    (d / "versions").write_text("libcudart.so.13 { global: *; };\n")
    so = str(d / "libcudart.so.13")
    subprocess.run(["gcc", "-std=gnu11", "-O1", "-shared", "-fPIC", "-I", os.path.join(CUDA, "include"), "-Wl,-soname,libcudart.so.13",
                    f"-Wl,--version-script={d / 'versions'}", os.path.join(HERE, "fake_cudart.c"), "-o", so], check=True)
    tables = {n: (f.k, f.s, f.dim, [int(v) for row in f.table() for v in row]) for n, f in W.FAMILIES.items()}
    prelude = PRELUDE.format(fake=so, lib=capi.LIB_PATH, tables=tables)

    def run(body):
        p = subprocess.run([sys.executable, "-c", prelude + body], capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, (p.returncode, p.stdout, p.stderr)
    return run


def test_tables_outlive_their_copy(host):
    # a copy from pageable memory may read its source until the stream has been waited for
    host("""
for name, r, steps in (("triangle", 8, 5), ("carpet", 8, 1), ("carpet", 10, 3), ("menger", 6, 1)):
    h = handle(name, r)
    assert step(h, steps, stream=0x70) == 0 and step(h, steps, stream=0x70) == 0
    assert not log("source changed", clear=False), name
    assert sliced(kernels()), name
b = c_void_p()
assert lib.fractal_batch_create(byref(b)) == 0
h = handle("triangle", 9)
assert lib.fractal_batch_add(b, h, c_void_p(A), c_void_p(B), c_int64(4), 8, 12, None) == 0
fake.fake_clear()
assert lib.fractal_batch_run(b, None) == 0
assert not log("source changed", clear=False) and sliced(kernels())
""")


def test_a_batch_readies_its_handles(host):
    # the allocation-free step and captured generations need tables that only earlier calls can build
    host("""
b, h = c_void_p(), handle("triangle", 9)
assert lib.fractal_batch_create(byref(b)) == 0
assert lib.fractal_batch_add(b, h, c_void_p(A), c_void_p(B), c_int64(4), 8, 12, None) == 0
assert lib.fractal_batch_run(b, None) == 0
assert sliced(kernels())
assert step(h, 3, fn="fractal_step_noalloc") == 0, lib.fractal_last_error()
fake.fake_capturing(1)
fake.fake_clear()
assert step(h, 1) == 0 and not log("malloc", clear=False) and len(kernels()) == 1
""")


def test_copies_come_before_generations(host):
    # an instance may start from what one of no generations copies, and overwrite what one of a single generation reads
    host("""
b, h = c_void_p(), handle("triangle", 9)
assert lib.fractal_batch_create(byref(b)) == 0
for n, src, dst in ((4, A, B), (0, A + (1 << 20), A), (1, B, B + (1 << 20))):
    assert lib.fractal_batch_add(b, h, c_void_p(src), c_void_p(dst), c_int64(n), 8, 12, None) == 0
assert lib.fractal_batch_run(b, None) == 0
order = ["copy" if "copy_normalise" in x else "sliced" if "resident" in x else "tiles" if "step_" in x else "" for x in kernels()]
assert [x for x in order if x] == ["copy", "tiles", "sliced"], order
""")


def test_box_words_are_kept_only_when_filled(host):
    # a call that cannot fill the packed box's arrays keeps none of them: one of the next calls fills them
    host("""
for name, r, steps, rule in (("carpet", 5, 3, (8, 12)), ("menger", 4, 1, (32, 48))):
    for call, after in (("cudaMemsetAsync", 0), ("launch", 0), ("cudaStreamSynchronize", 0), ("cudaMalloc", 0)):
        h = handle(name, r)
        assert step(h, 0, rule=rule, fn="fractal_bb_step") == 0        # builds the row kernels' tables
        held = fake.fake_held()
        fake.fake_clear()
        fake.fake_fail(call.encode(), after)
        step(h, steps, rule=rule, fn="fractal_bb_step")
        for _ in range(20):
            assert step(h, steps, rule=rule, fn="fractal_bb_step") == 0, lib.fractal_last_error()
        names = kernels()
        filled = [i for i, x in enumerate(names) if "bb_member" in x]
        assert filled and any("bb_words" in x for x in names[filled[-1]:]), (name, call, names)
        assert not any("bb_words" in x for x in names[:filled[-1]]), (name, call, names)
        assert step(h, 1 if steps > 1 else 2, rule=rule, fn="fractal_bb_step") == 0
        assert lib.fractal_destroy(h) == 0
assert fake.fake_held() == 0, fake.fake_held()
""")


def test_packed_boxes_need_no_scratch(host):
    # calls of several box generations hold packed boxes alone, and serve captured calls at any address
    host("""
for name, r, rule in (("carpet", 6, (8, 12)), ("menger", 4, (32, 48))):
    h, side, dim = handle(name, r), TABLES[name][1] ** r, TABLES[name][2]
    assert step(h, 3, rule=rule, fn="fractal_bb_step") == 0
    sizes = [int(x.split()[1]) for x in log("^malloc")]
    assert max(sizes) < side ** dim, (sizes, side ** dim)
    fake.fake_capturing(1)
    fake.fake_clear()
    for src, dst in ((A, B), (A + 3, B), (A, B + 5), (A + 1, B + 2)):
        assert step(h, 4, rule=rule, src=src, dst=dst, fn="fractal_bb_step") == 0, lib.fractal_last_error()
    assert not log("malloc", clear=False) and sum("bb_words" in x for x in kernels()) == 16
    fake.fake_capturing(0)
    lib.fractal_destroy(h)
""")


def test_sliced_again_when_memory_is_free_again(host):
    # calls that find no memory for the tables or the packed states run on the tile kernels; once there is memory,
    # one of the next calls has them
    host("""
for name, r, steps, room in (("carpet", 9, 4, 1 << 18), ("h_fractal", 10, 3, 1 << 18), ("h_fractal", 10, 3, 20 << 20)):
    h = handle(name, r)
    assert lib.fractal_get_tile_levels(h, byref(c_int())) == 0
    fake.fake_limit(fake.fake_held() + room)
    rc = step(h, steps)                       # (the ping-pong scratch may not fit either)
    assert not sliced([x for x in kernels() if "step_kernel" in x or "resident" in x]) and rc in (0, -3)
    fake.fake_limit(1 << 60)
    fake.cudaGetLastError()
    fake.fake_clear()
    assert all(step(h, steps) == 0 for _ in range(20))
    assert sliced([x for x in kernels() if "step_kernel" in x or "resident" in x]), (name, room)
    lib.fractal_destroy(h)
""")


def test_a_first_call_builds_what_it_uses(host):
    # calls that the tile kernels serve build no sliced tables; the others make one allocation for all they need
    host("""
def first(name, r, steps):
    h = handle(name, r)
    assert lib.fractal_get_tile_levels(h, byref(c_int())) == 0
    fake.fake_clear()
    assert step(h, steps) == 0
    mallocs, syncs = log("^malloc", clear=False), log("^sync", clear=False)
    names = kernels()
    assert lib.fractal_destroy(h) == 0
    return names, len(mallocs), len(syncs)
for name, r in (("carpet", 7), ("vicsek", 8), ("h_fractal", 6), ("candy", 5)):
    names, mallocs, syncs = first(name, r, 1)
    assert (sliced(names), mallocs, syncs) == (False, 0, 0), (name, names, mallocs)
for name, r, steps in (("triangle", 12, 1), ("carpet", 10, 1), ("carpet", 10, 4), ("menger", 7, 1), ("menger", 6, 3),
                       ("triangle", 8, 9)):
    names, mallocs, syncs = first(name, r, steps)
    assert (sliced(names), mallocs, syncs) == (True, 1, 1), (name, names, mallocs, syncs)
assert fake.fake_held() == 0
""")


def test_refused_allocations_are_tried_again_ever_later(host):
    # a refused allocation takes milliseconds: calls that run on the byte-wise kernels meanwhile do not try each time
    host("""
for name, r, fn, size in (("carpet", 7, "fractal_bb_step", 3 ** 14), ("h_fractal", 10, "fractal_step", 7 ** 10)):
    h = handle(name, r)
    assert step(h, 1, fn=fn) == 0
    # room for the byte-wise kernels' scratch alone, then for nothing more
    fake.fake_fail(b"cudaMalloc", 0)
    assert step(h, 3, fn=fn) == 0
    fake.fake_limit(fake.fake_held() + 1000)
    fake.cudaGetLastError()
    fake.fake_clear()
    assert all(step(h, 3, fn=fn) == 0 for _ in range(300))
    assert 1 <= len(log("^refused")) <= 6, name
    fake.fake_limit(1 << 60)
    assert all(step(h, 3, fn=fn) == 0 for _ in range(600))
    fake.fake_clear()
    assert step(h, 3, fn=fn) == 0
    assert any("bb_words" in x or "slice_" in x for x in kernels()), name
    lib.fractal_destroy(h)
""")


def test_a_single_call_does_not_pay_for_tables(host):
    # a handle's first single generation runs on the tile kernels unless the state is large or needs no packed state;
    # the second one, a call of several and the autotuner have the tables built
    host("""
def calls(name, r, *steps):
    h, out = handle(name, r), []
    for n in steps:
        fake.fake_clear()
        assert step(h, n) == 0
        out.append(sliced(kernels()))
    lib.fractal_destroy(h)
    return out
for name, r in (("carpet", 9), ("h_fractal", 8), ("menger", 6)):
    assert calls(name, r, 1, 1, 1) == [False, True, True], name
    assert calls(name, r, 1, 3) == [False, True], name
    assert calls(name, r, 3, 1) == [True, True], name
for name, r in (("carpet", 10), ("menger", 7), ("triangle", 14)):
    assert calls(name, r, 1) == [True], name
h = handle("carpet", 9)
assert lib.fractal_autotune(h, c_void_p(A), c_void_p(B), 8, 12, None, None) == 0
assert sliced(kernels())
""")


def test_a_few_generations_of_small_states(host):
    # two generations (3D: a few) of small states are a launch each of the tile kernels; a captured call takes what exists
    host("""
def call(h, n):
    fake.fake_clear()
    assert step(h, n) == 0, lib.fractal_last_error()
    return sliced(kernels())
for name, r, most in (("triangle", 10, 2), ("triangle", 12, 2), ("vicsek", 7, 2), ("vicsek", 10, 2), ("chandelier", 9, 2), ("menger", 2, 2),
                      ("triangle", 8, 1), ("carpet", 8, 1), ("full_square", 8, 1), ("menger", 3, 1), ("vicsek", 5, 1)):
    h = handle(name, r)
    assert [call(h, n) for n in (2, 3, 4, 10)] == [n > most for n in (2, 3, 4, 10)], (name, r)
    lib.fractal_destroy(h)
h = handle("triangle", 10)
assert call(h, 3)
fake.fake_capturing(1)
assert call(h, 2) and not log("malloc")
""")


def test_short_box_views_go_cell_by_cell(host):
    host("""
for name, r, tiles in (("menger", 4, False), ("carpet", 6, False), ("vicsek", 8, False), ("triangle", 12, True), ("h_fractal", 7, True)):
    h = handle(name, r)
    fake.fake_clear()
    assert lib.fractal_scatter_to_box(h, c_void_p(A), c_void_p(B), None) == 0
    assert lib.fractal_gather_from_box(h, c_void_p(A), c_void_p(B), None) == 0
    assert ["box_tiles" in x for x in kernels()] == [tiles, tiles], (name, r)
""")


def test_batches_of_two_short_generations(host):
    # one class of instances and two generations: a launch of the tile kernels each; more classes or generations go sliced
    host("""
def run(*instances):
    b = c_void_p()
    assert lib.fractal_batch_create(byref(b)) == 0
    for i, (name, r, n) in enumerate(instances):
        assert lib.fractal_batch_add(b, handle(name, r), c_void_p(A + (i << 28)), c_void_p(B + (i << 28)), c_int64(n), 8, 12, None) == 0
    fake.fake_clear()
    assert lib.fractal_batch_run(b, None) == 0
    names = [x for x in kernels() if "resident" in x or "step_" in x]
    lib.fractal_batch_destroy(b)
    return sliced(names), len(names)
assert run(("triangle", 12, 2), ("triangle", 12, 2)) == (False, 2)
assert run(("triangle", 10, 2), ("carpet", 6, 2), ("vicsek", 8, 2)) == (False, 6)
assert run(("triangle", 12, 3), ("triangle", 12, 2))[0]
assert run(("triangle", 12, 2), ("triangle", 4, 2), ("triangle", 5, 2))[0]
assert run(("triangle", 16, 2))[0]
""")


def test_settings_after_the_autotuner(host):
    # a setting given back to the library is the library's again, whatever the autotuner had chosen; one set by the
    # caller asks for the tile kernels
    host("""
def tuned():
    h = handle("carpet", 8)
    assert lib.fractal_autotune(h, c_void_p(A), c_void_p(B), 8, 12, None, None) == 0
    return h
def goes_sliced(h, n=4):
    fake.fake_clear()
    assert step(h, n) == 0
    return sliced(kernels())
assert goes_sliced(tuned()) and goes_sliced(handle("carpet", 8))
for fn, back, own in ((lib.fractal_set_tile_levels, -1, 3), (lib.fractal_set_pipeline_stages, -1, 3)):
    h = tuned()
    assert fn(h, back) == 0 and goes_sliced(h)
    assert fn(h, own) == 0 and not goes_sliced(h)
    assert fn(h, back) == 0 and goes_sliced(h)
h = tuned()
assert lib.fractal_set_tile_levels(h, -1) == 0 and lib.fractal_set_pipeline_stages(h, -1) == 0 and goes_sliced(h)
""")


def test_streams_wait_only_where_buffers_are_shared(host):
    # one handle on two streams: single generations do not wait for the other stream, calls of several wait for calls
    # of several alone, box calls never for compact ones
    host("""
def call(h, fn, n, stream):
    fake.fake_clear()
    assert step(h, n, stream=stream, fn=fn, rule=rule) == 0
    waits = log("^wait", clear=False)
    return len(waits), any("slice_" in x or "bb_words" in x for x in kernels())
for name, r, rule in (("carpet", 10, (8, 12)), ("h_fractal", 8, (8, 12)), ("menger", 6, (32, 48))):
    h, step1, box1 = handle(name, r), ("fractal_step", 1), ("fractal_bb_step", 1)
    step3, box3 = ("fractal_step", 3), ("fractal_bb_step", 3)
    calls = [step1, step3] + ([box1, box3] if name == "menger" else [box3] if name == "h_fractal" else [])
    for c in calls:
        for _ in range(2):
            call(h, *c, 0x10)
        assert call(h, *c, 0x10)[1], (name, c)
    fake.fake_events_pending(1)
    for c in calls:
        waits, packed = call(h, *c, 0x20)
        assert (waits, packed) == ((0, False) if c[1] == 1 else (1, True)), (name, c, waits, packed)
    fake.fake_events_pending(0)
    for c in calls:
        assert call(h, *c, 0x20) == (1, True), (name, c)
    lib.fractal_destroy(h)
""")


def test_armed_calls_with_grid_barriers_stay_sliced(host):
    # the failure-detection hook reaches the sliced step's grid barriers; calls without one go to the tile kernels
    host("""
for name, r, n, barrier in (("carpet", 8, 6, True), ("h_fractal", 10, 4, True), ("menger", 6, 5, True), ("triangle", 4, 6, False),
                            ("carpet", 10, 1, False), ("triangle", 14, 1, False)):
    h = handle(name, r)
    for armed in (False, True, False):
        assert not armed or lib.fractal_test_arm_timeout(h, 16, 256) == 0
        fake.fake_clear()
        assert step(h, n) == 0
        assert sliced([x for x in kernels() if "nbr" not in x]) == (barrier or not armed), (name, armed)
    lib.fractal_destroy(h)
""")
