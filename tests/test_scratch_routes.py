"""Which kernel a sketch takes and what scratch it touches, on the host side alone: libsk runs over a CUDA runtime
without a GPU (tests/fake_cudart.c, preloaded in a child process) that counts launches and allocations and can be
told that a stream is being captured, that earlier work is still running, or that an allocation fails. Kernels are
not run, so nothing here says anything about results."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
sys.path.insert(0, %r)
from paper_2606_20195_gb300 import sk
fake = ctypes.CDLL(None)
def var(name, t=ctypes.c_int): return t.in_dll(fake, name)
capturing, busy, most = var("fake_capturing"), var("fake_busy"), var("fake_max", ctypes.c_ulonglong)
kernels, coop, mallocs, frees = var("fake_kernels"), var("fake_coop"), var("fake_mallocs"), var("fake_frees")
GATHER, BAR = 7, 256
A, Y, ST = 1 << 20, 1 << 21, 64  # addresses that nothing reads
SMALL = dict(d=256, m=16384, k=4), 16      # one launch (short slices), else one slice per chunk
GATH = dict(d=4096, m=65536, k=1), 128     # gather kernel, else the tile kernel with one slice per chunk
REG16 = dict(d=512, m=4000, k=4), 64       # register kernel for a 16-bit A, else the tile kernel
BOTH = dict(d=4096, m=1 << 22, k=1), 64    # gather kernel, else the tile kernel with chunk totals too
def totals(case, chunks): return 4 * chunks * case[0]["d"] * case[1]
def apply(p, n, st=ST, a_type=0, lda=None):
    c0, k0 = coop.value, kernels.value
    if a_type: sk.sk_apply_typed(p.handle, A, a_type, lda or n, n, Y, st)
    else: sk.sk_apply(p.handle, A, lda or n, n, Y, st)
    return p.get(sk.SK_PARAM_LAST_KERNEL), coop.value - c0, kernels.value - k0
def plan(case, rule=1, **kw): return sk.Plan(case[0]["d"], case[0]["m"], case[0]["k"], rule, 1, **kw)
def held(p): return p.get(sk.SK_PARAM_SCRATCH_BYTES)
TILE, REG, GLOBAL = sk.SK_KERNEL_TILE, sk.SK_KERNEL_REGISTER, sk.SK_KERNEL_GLOBAL
""" % ROOT


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2606_20195_gb300 import _build
    _build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-Wno-builtin-declaration-mismatch", "-o", lib,
                    os.path.join(HERE, "fake_cudart.c")], check=True)

    def go(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE + body], capture_output=True, text=True,
                           env={**os.environ, "LD_PRELOAD": lib, "CUDA_VISIBLE_DEVICES": ""})
        assert r.returncode == 0, r.stdout + r.stderr
    return go


def test_routes(run):
    run("""
p = plan(SMALL); assert apply(p, 16) == (TILE, 1, 0) and held(p) == 4 + BAR + totals(SMALL, 4), held(p)
p = plan(GATH); assert apply(p, 128)[0] == GATHER and held(p) == 4 + BAR + totals(GATH, 8), held(p)
p = plan(REG16); assert apply(p, 64, a_type=1)[0] == REG and held(p) == 4 + BAR + totals(REG16, 1), held(p)
p = plan(BOTH); assert apply(p, 64)[0] == GATHER and held(p) == 4 + totals(BOTH, 8), held(p)
""")


def test_capture_takes_no_scratch_that_a_later_call_may_free(run):
    # A graph keeps the addresses of its launches. Sketches that need no chunk totals must not put totals into
    # one, even where the plan has them already: a later, larger call frees the buffer.
    run("""
for case, n, t in ((SMALL, 16, 0), (GATH, 128, 0), (REG16, 64, 1)):
    p = plan(case); first = apply(p, n, a_type=t); before = held(p)
    capturing.value = 1
    assert apply(p, n, a_type=t) == (TILE, 0, 1)
    assert held(p) == before
    capturing.value = 0
    assert apply(p, n, a_type=t) == first
p = plan(BOTH); first = apply(p, 64); capturing.value = 1
assert apply(p, 64) == first  # (needs the plan's totals in either form)
""")


def test_another_streams_totals_are_left_alone(run):
    run("""
for case, n, t in ((SMALL, 16, 0), (GATH, 128, 0), (REG16, 64, 1)):
    p = plan(case); fast = apply(p, n, 64, t); busy.value = 1
    assert apply(p, n, 64, t) == fast            # the same stream: in order
    assert apply(p, n, 128, t) == (TILE, 0, 1)   # another one, while the first may be running
    assert apply(p, n, 64, t) == fast
    busy.value = 0
    assert apply(p, n, 128, t) == fast; busy.value = 1
    assert apply(p, n, 64, t) == (TILE, 0, 1); busy.value = 0
""")


def test_a_failed_allocation_takes_the_form_that_needs_less(run):
    run("""
most.value = 1 << 15  # cudaMalloc of more than this fails
for case, n, t in ((SMALL, 16, 0), (GATH, 128, 0), (REG16, 64, 1)):
    p = plan(case)
    assert apply(p, n, a_type=t) == (TILE, 0, 1) and held(p) == 4
WIDE = dict(d=8190, m=65536, k=3), 257  # gather kernel, else the global kernel, in passes with smaller totals
p = plan(WIDE); most.value = 0; assert apply(p, 257)[0] == GATHER; need = held(p) - 4
p = plan(WIDE); most.value = need - 1
assert apply(p, 257)[0] == GLOBAL and 4 < held(p) < 4 + need
""")


def test_short_chunks_need_no_large_totals(run):
    # Totals are d x n floats for every chunk: with the chunk length of the paper's per-element scheme (1) they
    # would be 17 TB here. What a plan holds for speed stays below A's own size in FP32.
    run("""
for R, t in ((1, 0), (1, 1), (7, 0), (64, 1), (256, 0), (1000, 1)):
    p = sk.Plan(1024, 65536, 1 if t == 0 else 4, 1, 1, chunk_rows=R)
    assert apply(p, 64, a_type=t)[0] == TILE and held(p) <= 4 + BAR + 4 * 65536 * 64, (R, t)
p = sk.Plan(4096, 1 << 22, 1, 1, 1, chunk_rows=256)
assert apply(p, 64)[0] == TILE and held(p) == 4
for R, case, n, t, kern in ((0, GATH, 128, 0, GATHER), (8192, BOTH, 64, 0, TILE), (1 << 17, BOTH, 64, 0, GATHER),
                            (2048, REG16, 64, 1, REG), (200, REG16, 64, 1, TILE)):
    p = plan(case, chunk_rows=R)
    assert apply(p, n, a_type=t)[0] == kern, (R, case)
""")


def test_gather_kernel_leaves_tall_sketches_to_others(run):
    # The gather kernel's work grows with d n; the kernels taken otherwise make k n additions a row whatever d.
    run("""
for d, m, k, n, want in ((32768, 1 << 20, 2, 33, False), (262144, 1 << 20, 2, 33, False), (1 << 20, 1 << 20, 8, 33, False),
                         (16384, 1 << 18, 4, 65, False), (16384, 1 << 22, 4, 65, True), (8192, 32768, 4, 33, True),
                         (65536, 1 << 20, 2, 28, False), (2048, 1 << 20, 2, 28, True), (4096, 1 << 22, 2, 24, False),
                         (15000, 1 << 17, 4, 100, False), (8192, 1 << 17, 4, 100, True), (1024, 1 << 17, 1, 512, False),
                         (1024, 1 << 19, 1, 512, True), (4096, 40000, 4, 128, False), (4096, 1 << 17, 4, 128, True),
                         (8192, 1 << 17, 3, 1537, False), (4096, 1 << 17, 3, 1537, True), (1024, 40000, 3, 5001, False),
                         (2048, 65536, 1, 257, False), (2048, 1 << 18, 1, 257, True), (2048, 40000, 1, 130, False)):
    p = sk.Plan(d // k * k, m, k, 1, 1)
    assert (apply(p, n)[0] == GATHER) == want, (d, m, k, n)
""")


def test_optional_totals_are_given_back(run):
    # The totals a sketch can do without must not stand in the way of scratch that a later call needs: under the
    # limit that sk_solve or sk_apply_host needs by itself, and where the device's memory is short.
    run("""
for case, n in ((SMALL, 16), (GATH, 128)):
    alone = plan(case)
    sk.sk_solve_sketched(alone.handle, Y, n + 1, n, Y, ST); need = held(alone)
    p = plan(case)
    fast = apply(p, n)
    p.set(sk.SK_PARAM_SCRATCH_LIMIT, need + 4 + 1000)  # room for the solve's scratch, not for both
    f0 = frees.value
    sk.sk_solve(p.handle, A, n, n, A, Y, ST)
    assert held(p) <= need + 4 and frees.value == f0 + 1
    assert apply(p, n) == (TILE, 0, 1) and held(p) == need + 4
    p.set(sk.SK_PARAM_SCRATCH_LIMIT, 0)
    assert apply(p, n) == fast
    p = plan(case); apply(p, n)
    tile = 4 * case[0]["m"] * n; y = 2 * case[0]["d"] * n
    p.set(sk.SK_PARAM_SCRATCH_LIMIT, 4 + 2 * tile + y)
    out = ctypes.create_string_buffer(y)
    sk.sk_apply_host(p.handle, A, n, n, ctypes.addressof(out), ST)
    assert held(p) == 4 + 2 * tile + y
""")


def test_small_sketches_leave_room_beside_them(run):
    # A one-launch sketch waits at a grid barrier, so its CTAs must all be resident: over half of the GPU's 152, two
    # calls on two streams run one after the other. Small ones are as fast on half of them.
    run("""
grid = var("fake_grid", ctypes.c_uint)
for (m, n, d, k), half in (((16384, 16, 256, 4), True), ((20000, 1, 256, 4), True), ((3000, 12, 4096, 2), True),
                           ((60000, 20, 320, 8), False), ((30000, 32, 1024, 1), False)):
    p = sk.Plan(d, m, k, 1, 1)
    assert apply(p, n) == (TILE, 1, 0)
    assert (grid.value <= 76) == half and grid.value >= 38, (m, n, grid.value)
""")


def test_totals_that_were_not_zeroed_are_not_kept(run):
    run("""
fails = var("fake_memset_fails")
for case, n, t in ((GATH, 128, 0), (REG16, 64, 1)):
    p = plan(case); fails.value = 1
    try: apply(p, n, a_type=t)
    except sk.SkError: pass  # (zeroing Y fails too)
    fails.value = 0
    assert held(p) == 4
    assert apply(p, n, a_type=t)[0] in (GATHER, REG)
""")
