"""The library's host code without a GPU: what it allocates, frees and keeps, and launches.

A child process runs libpce.so on a CUDA runtime of host memory (fake_cudart.cpp) that counts
work as pending until its stream or the device is synchronised.
"""
import os
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
fake = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
sys.path.insert(0, sys.argv[2])
import paper_1604_04374_gb300.pce as pce
lib = pce.load_library()
P, SZ = ctypes.c_void_p, ctypes.c_size_t
for f in ("fake_live_bytes", "fake_kept_bytes"):
    getattr(fake, f).restype = SZ
fake.fake_set_capacity.argtypes = [SZ]
fake.fake_fail_alloc.argtypes = [ctypes.c_longlong]
fake.cudaMalloc.argtypes = [ctypes.POINTER(P), SZ]
fake.fake_launch.restype = ctypes.c_char_p
fake.fake_launch.argtypes = [ctypes.c_int, P, P]
S1, S2 = 0x1000, 0x2000   # streams

def dmalloc(floats):
    p = P()
    assert fake.cudaMalloc(ctypes.byref(p), 4 * floats) == 0
    ctypes.memset(p, 0, 4 * floats)
    return p.value

def create(shape, m, flags=0, stream=S1, sep=False):
    \"\"\"(status, handle) of a plan of zero windows.\"\"\"
    n = 1
    for d in shape:
        n *= d
    out, shp, h = P(), (ctypes.c_int64 * len(shape))(*shape), dmalloc(m * n)
    if sep:
        st = lib.pce_plan_create_separable(ctypes.byref(out), shp, m, dmalloc(m * shape[0]), dmalloc(m * shape[1]), h,
                                           flags, P(stream))
    else:
        st = lib.pce_plan_create(ctypes.byref(out), len(shape), shp, m, dmalloc(m * n), h, flags, P(stream))
    return st, out.value

def same(*pairs):
    for a, b in zip(pairs[::2], pairs[1::2]):
        if a != b:
            raise AssertionError(f"{a} != {b} (last error: {lib.pce_last_error_string()})")

def pool():
    return fake.fake_live_bytes() - base

def launches():
    d, smem, out = (ctypes.c_uint * 6)(), SZ(), []
    for i in range(fake.fake_launches()):
        name = fake.fake_launch(i, d, ctypes.byref(smem)).decode()
        out.append((name, tuple(d[:3]), tuple(d[3:])))
    return out
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_1604_04374_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfakecudart.so")
    cuda = os.path.dirname(os.path.dirname(build._nvcc()))
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", so], check=True)

    def run(body):
        res = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body), so, ROOT], timeout=300,
                             stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
        assert res.returncode == 0, res.stdout.decode(errors="replace")[-4000:]

    return run


@pytest.mark.parametrize("shape", [(4096,), (16384,), (256, 256)])
def test_a_plan_that_cannot_wait_keeps_its_memory(child, shape):
    """A device synchronisation is an error while a stream of the device is captured.  A plan
    destroyed then, its work pending, says so, and none of its memory goes back before a later
    call has waited."""
    child(f"""
    shape = {shape}
    n = shape[0] * (shape + (1,))[1]
    u, y = dmalloc(n), dmalloc(n)
    st, plan = create(shape, 4)
    st2, other = create(shape, 4)
    same(st, 0, st2, 0)
    base = fake.fake_live_bytes()
    same(lib.pce_apply(P(plan), P(u), P(y), 1, P(S2)), 0)
    fake.fake_set_capturing(1)
    same(lib.pce_plan_destroy(P(plan)), pce.PCE_ERR_CUDA)
    same(fake.fake_unordered_frees(), 0, pool(), 0, fake.fake_pending(), 1)
    fake.fake_set_capturing(0)
    same(lib.pce_plan_destroy(P(other)), 0)   # waits: both plans' memory goes back
    freed = -pool()
    same(fake.fake_unordered_frees(), 0)
    # the same when the memory is asked for
    st, plan = create(shape, 4)
    base = fake.fake_live_bytes()
    same(lib.pce_apply(P(plan), P(u), P(y), 1, P(S2)), 0)
    fake.fake_set_capturing(1)
    same(lib.pce_plan_destroy(P(plan)), pce.PCE_ERR_CUDA, lib.pce_release_memory(), pce.PCE_ERR_CUDA, pool(), 0)
    fake.fake_set_capturing(0)
    same(lib.pce_release_memory(), 0)
    same(2 * -pool(), freed, fake.fake_unordered_frees(), 0, fake.fake_kept_bytes(), 0)
    """)


def test_a_handle_is_destroyed_once(child):
    """Plan.close() and Batch.close() give their handle up also where the call fails: a second
    close, and the object's end, leave it alone."""
    child("""
    st, plan = create((256, 256), 4)
    same(st, 0)
    u, y = dmalloc(65536), dmalloc(65536)
    obj = object.__new__(pce.Plan)
    obj.handle = plan
    same(lib.pce_apply(P(plan), P(u), P(y), 1, P(S2)), 0)
    base = fake.fake_live_bytes()
    fake.fake_set_capturing(1)
    try:
        obj.close()
    except pce.PceError as e:
        same(e.status, pce.PCE_ERR_CUDA)
    else:
        raise AssertionError("the destroy did not fail")
    same(obj.handle, None)
    fake.fake_set_capturing(0)
    obj.close()
    same(pool(), 0)
    same(lib.pce_release_memory(), 0, fake.fake_unordered_frees(), 0)
    assert pool() < 0
    del obj
    batch = object.__new__(pce.Batch)
    batch.handle, batch._keep = 1, []
    pce.pce_batch_destroy = lambda handle: (_ for _ in ()).throw(pce.PceError(4, "fails"))
    try:
        batch.close()
    except pce.PceError:
        pass
    same(batch.handle, None)
    batch.close()
    """)


@pytest.mark.parametrize("shape,m,flags,sep", [((512, 64), 3, 0, True), ((1024, 32), 2, 0, True),
                                               ((256, 64), 2, 0, False), ((1024, 64), 2, "SECTIONED", False),
                                               ((2048, 16), 2, "LOWP_STORAGE", False), ((2048,), 3, 0, False),
                                               ((32768,), 3, 0, False)])
def test_a_failed_creation_frees_in_order(child, shape, m, flags, sep):
    """Every allocation of a plan's creation fails in turn: the creation reports it, what it
    had allocated goes back, and only after its stream's work."""
    child(f"""
    shape, m, sep = {shape}, {m}, {sep}
    flags = pce.PCE_FLAG_{flags} if {flags!r} else 0
    base0 = fake.fake_live_bytes()
    st, plan = create(shape, m, flags, S1, sep)
    same(st, 0, lib.pce_plan_destroy(P(plan)), 0)
    inputs = fake.fake_live_bytes() - base0   # create()'s own
    for n in range(200):
        base = fake.fake_live_bytes()
        fake.fake_fail_alloc(n + (3 if sep else 2))
        st, plan = create(shape, m, flags, S1, sep)
        fake.fake_fail_alloc(-1)
        fake.cudaGetLastError()
        if st == 0:
            break
        assert st in (pce.PCE_ERR_OOM, pce.PCE_ERR_CUDA), st
        same(plan, None, pool(), inputs, fake.fake_unordered_frees(), 0)
    assert 3 < n < 199, n
    same(lib.pce_plan_destroy(P(plan)), 0, fake.fake_unordered_frees(), 0)
    """)


@pytest.mark.parametrize("call", ["plan", "batch", "autotune", "svd", "projection_1d", "projection_2d"])
def test_what_the_pool_keeps_serves_every_allocation(child, call):
    """Memory of closed plans serves the library's next allocation, of whatever kind, where the
    device has no other; where there is none at all the call is refused, and its refusal is not
    reported again by the next one."""
    child(f"""
    call = {call!r}
    st, held = create((1024, 1024), 1)
    same(st, 0)
    keep = [create((65536,), 2)[1] for _ in range(2)]
    n = 1024 * 1024
    u, y0, y1, T, h, w, w2 = (dmalloc(n) for _ in range(7))
    task = (pce.PceTask * 2)(*(pce.PceTask(k, u, y, 1, 0, 0) for k, y in zip(keep, (y0, y1))))
    shape, out = (ctypes.c_int64 * 1)(8192), P()

    def run():
        \"\"\"Whether memory ran out.\"\"\"
        if call == "plan":
            st = lib.pce_plan_create(ctypes.byref(out), 1, shape, 32, P(u), P(T), 0, P(S1))
        elif call == "batch":
            st = lib.pce_batch_create(ctypes.byref(out), task, 2, 2)
        elif call == "autotune":
            st = lib.pce_plan_autotune(P(keep[0]), 1, None, P(S1))
        elif call == "svd":
            st = lib.pce_construct_svd_1d(P(T), 1024, 8, 10, 2, 0, P(h), P(w), None, P(S1))
        elif call == "projection_1d":
            st = lib.pce_construct_projection_1d(P(T), 1024, 8, P(h), P(w), P(S1))
        else:
            st = lib.pce_construct_projection_2d(P(T), 32, 32, 16, 16, 2, 2, P(h), P(w), P(w2), P(S1))
        # (the windows are zero here: a projection that got its memory ends at its Gram matrix)
        assert st != pce.PCE_ERR_INVALID or b"singular" in lib.pce_last_error_string()
        return st != 0 and b"out of memory" in lib.pce_last_error_string()

    same(lib.pce_release_memory(), 0)
    fake.fake_set_capacity(fake.fake_live_bytes() + 1024)   # nothing left for it
    for _ in range(2):
        same(run(), True, fake.cudaGetLastError(), 0)
    kept = fake.fake_kept_bytes()
    same(lib.pce_plan_destroy(P(held)), 0)
    assert fake.fake_kept_bytes() > kept + (4 << 20)        # its memory stays in the pool
    same(run(), False, fake.cudaGetLastError(), 0, fake.fake_unordered_frees(), 0)
    """)


@pytest.mark.parametrize("shape", [(64, 1024), (256, 512), (512, 512), (1024, 512), (1024, 1024), (2048, 256)])
def test_column_splits_stay_within_one_wave(child, shape):
    """The CTAs that share a column tile's terms are doubled while all of them are resident at
    once, by the threads and shared memory of the kernel that runs."""
    child(f"""
    shape, m = {shape}, 16
    st, plan = create(shape, m)
    same(st, 0)
    u, y = (dmalloc(shape[0] * shape[1]) for _ in range(2))
    splits = 0
    for cv in (0, 1) if shape[0] >= 512 else (0,):
        same(lib.pce_plan_set_tuning(P(plan), 0, cv, 0), 0)
        fake.fake_clear_launches()
        same(lib.pce_apply(P(plan), P(u), P(y), 1, P(S1)), 0, lib.pce_apply_adjoint(P(plan), P(u), P(y), 1, P(S1)), 0)
        d, smem, found = (ctypes.c_uint * 6)(), SZ(), 0
        for i in range(fake.fake_launches()):
            name = fake.fake_launch(i, d, ctypes.byref(smem)).decode()
            if "cols" not in name:
                continue
            found += 1
            resident = min(2048 // d[3], 233472 // (smem.value + 1024))
            ctas = d[0] * d[1] * d[2]
            splits += d[2] > 1
            assert d[2] == 1 or ctas <= 152 * resident, (cv, name, list(d), smem.value, resident)
        same(found, 2)
    assert splits > 0
    """)


def test_dense_forward_splits_where_its_rounds_are_full(child):
    """Eight or four CTAs share a column tile's terms where the rounds are full enough and the
    chain is long enough for the length, and all CTAs are resident at once; none otherwise."""
    child("""
    for ny, cases in ((256, ((4, 1, 1), (5, 1, 1), (7, 1, 1), (8, 1, 8), (8, 2, 8), (8, 4, 1), (9, 1, 1), (11, 2, 8),
                             (12, 2, 8), (16, 1, 8), (16, 4, 1), (17, 1, 8), (24, 1, 8), (28, 4, 4), (32, 8, 1))),
                      (128, ((4, 1, 1), (8, 8, 8), (8, 16, 4), (9, 1, 8), (9, 16, 4), (10, 16, 4), (12, 4, 8), (16, 24, 1)))):
        for m, batch, split in cases:
            st, plan = create((ny, ny), m)
            same(st, 0)
            u, y = (dmalloc(ny * ny * batch) for _ in range(2))
            fake.fake_clear_launches()
            same(lib.pce_apply(P(plan), P(u), P(y), batch, P(S1)), 0)
            got = [grid[2] for name, grid, block in launches() if "k_cols_fwd" in name]
            same((ny, m, batch, got), (ny, m, batch, [split]))
            same(lib.pce_plan_destroy(P(plan)), 0)
    """)
