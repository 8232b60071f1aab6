"""Host side of the library on a fake CUDA runtime (fake_cudart.c): what is
allocated, which launches are made and with which arguments, and what a call answers
when the runtime refuses one.  Each scenario runs in a child process.
"""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(ROOT, "paper_2602_05255_gb300", "liblrugb.so")

PRELUDE = r"""
import ctypes as C
fake = C.CDLL(None)
lib = C.CDLL(LIB)
for f, r, a in (("fake_alloc_limit", None, [C.c_size_t]), ("fake_total_limit", None, [C.c_size_t]),
                ("fake_refuse_launch", None, [C.c_char_p]), ("fake_watch", None, [C.c_char_p, C.c_int]),
                ("fake_launch_name", C.c_char_p, [C.c_int]), ("fake_launch_arg", C.c_void_p, [C.c_int]),
                ("fake_alloc_bytes", C.c_size_t, [C.c_int])):
    getattr(fake, f).restype, getattr(fake, f).argtypes = r, a
DET, PF, F64, C128, F32, C64, OK = 0, 1, 0, 1, 2, 3, 0
SIZE = {F64: 8, C128: 16, F32: 4, C64: 8}

class Cfg(C.Structure):
    _fields_ = [("kind", C.c_int32), ("dtype", C.c_int32), ("walkers", C.c_int64), ("n", C.c_int32),
                ("n_per_walker", C.c_void_p), ("k", C.c_int32), ("k_per_walker", C.c_void_p),
                ("delay", C.c_int32), ("flush", C.c_int32), ("device", C.c_int32), ("arith", C.c_int32),
                ("tile_chunks", C.c_int32), ("refresh", C.c_int32)]

class Operand(C.Structure):
    _fields_ = [("dense", C.c_void_p), ("idx", C.c_void_p), ("onehot_mask", C.c_uint32)]

PTR = C.c_void_p(4096)    # a device pointer: nothing reads through it

def create(kind=DET, dtype=F64, W=1024, n=128, k=1, delay=4, device=0, refresh=0, flush=0):
    cfg = Cfg(kind=kind, dtype=dtype, walkers=W, n=n, k=k, delay=delay, device=device, refresh=refresh, flush=flush)
    h = C.c_void_p()
    assert lib.lru_create(C.byref(cfg), C.byref(h)) == OK
    return h

def init(h, kind=DET):
    return (lib.lru_init_pf if kind == PF else lib.lru_init_det)(h, PTR, PTR, PTR)

def propose(h):
    o = Operand(4096, None, 0)
    return lib.lru_propose_det(h, C.byref(o), C.byref(o), PTR, PTR)

def accept(h):
    return lib.lru_accept(h, None)

def names():
    return [fake.fake_launch_name(i).decode() for i in range(fake.fake_launches())]

def refused():
    return [n for i, n in enumerate(names()) if not fake.fake_launch_ok(i)]

def sizes(ok=None):
    return [fake.fake_alloc_bytes(i) for i in range(fake.fake_allocs()) if ok is None or fake.fake_alloc_ok(i) == ok]
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not os.path.exists(LIB):
        import __graft_entry__
        __graft_entry__.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfakecudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)

    def go(body):
        r = subprocess.run([sys.executable, "-c", f"LIB = {LIB!r}\n" + PRELUDE + textwrap.dedent(body)],
                           env={**os.environ, "LD_PRELOAD": so}, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr

    return go


def test_flush_of_handles_on_two_devices(run):
    """The shared-memory limit of a kernel belongs to the device: the second one is not left with the first's."""
    run("""
        hs = [create(n=130, device=d) for d in (0, 1)]     # the kernel of ragged rows, which no elimination uses
        for h in hs:
            assert init(h) == OK
            for _ in range(5):
                assert propose(h) == OK and accept(h) == OK, (refused())
        assert any("k_oz_gemm" in x for x in names()) and not refused()
    """)


@pytest.mark.parametrize("flush", [0, 6])
def test_flush_that_is_not_launched_keeps_its_slots(run, flush):
    """No launch that resets tau after a refused product, and no update on top of it before an init."""
    run(f"""
        h = create(flush={flush})
        assert init(h) == OK
        assert propose(h) == OK and accept(h) == OK
        n = sum("k_flush_finish" in x for x in names())
        assert n == 1
        fake.fake_refuse_launch(b"k_oz_gemm")
        assert propose(h) == OK and accept(h) == 2
        assert sum("k_flush_finish" in x for x in names()) == n
        fake.fake_refuse_launch(b"")
        assert propose(h) == 4 and lib.lru_flush_delayed(h, None) == 4
        assert init(h) == OK and propose(h) == OK and accept(h) == OK
        assert sum("k_flush_finish" in x for x in names()) == n + 1
    """)


@pytest.mark.parametrize("dtype", [0, 1])
def test_standalone_calls_see_a_wait_that_gives_up(run, dtype):
    """The products of the calls without a handle get an error word, inside the call's own workspace."""
    run(f"""
        slogdet, grad = lib.lru_slogdet_batched, lib.lru_slogdet_backward
        slogdet.argtypes = [C.c_int32, C.c_int64, C.c_int32] + [C.c_void_p] * 4
        grad.argtypes = [C.c_int32, C.c_int64, C.c_int32] + [C.c_void_p] * 6
        for watch, at, call in ((b"k_oz_gemm", 7, lambda: slogdet({dtype}, 4, 130, PTR, PTR, PTR, None)),
                                (b"k_oz_gemm", 7, lambda: grad({dtype}, 4, 130, PTR, PTR, None, None, PTR, None)),
                                (b"k_slog_grad", 6, lambda: grad({dtype}, 4, 130, PTR, PTR, None, None, PTR, None))):
            fake.fake_reset()
            fake.fake_watch(watch, at)
            assert call() == OK
            got = {{fake.fake_launch_arg(i) for i, x in enumerate(names()) if watch.decode() in x}}
            assert len(got) == 1 and None not in got and len(sizes()) == 1, (watch, got)
    """)


@pytest.mark.parametrize("kind,dtype,n,per_sm", [("DET", "F64", 100, 2), ("DET", "C64", 100, 2), ("DET", "F32", 600, 2),
                                                 ("PF", "F64", 64, 4), ("PF", "F64", 1024, 4), ("PF", "F64", 1026, 2),
                                                 ("PF", "C128", 64, 2), ("PF", "C128", 1024, 2), ("PF", "F32", 64, 2)])
def test_elimination_slots_are_those_the_kernel_fills(run, kind, dtype, n, per_sm):
    """Copies of the kernels with a CTA per matrix: what a handle and the standalone Pfaffian allocate."""
    run(f"""
        slots = {per_sm} * 152 * {n} * {n} * SIZE[{dtype}]
        h = create(kind={kind}, dtype={dtype}, W=1000, n={n}, delay=0, refresh=1)
        fake.fake_reset()
        assert lib.lru_refresh_from_scratch(h, PTR, None, PTR) == OK and sizes() == [slots], (sizes(), slots)
        if {kind} == PF:
            f = lib.lru_slogpf_batched
            f.argtypes = [C.c_int32, C.c_int64, C.c_int32] + [C.c_void_p] * 4
            fake.fake_reset()
            assert f({dtype}, 1000, {n}, PTR, PTR, PTR, None) == OK and sizes() == [slots]
            # where four copies per SM are not to be had, two still serve
            fake.fake_reset()
            fake.fake_alloc_limit(2 * 152 * {n} * {n} * SIZE[{dtype}])
            assert f({dtype}, 1000, {n}, PTR, PTR, PTR, None) == OK
    """)


def test_refused_flush_workspace_is_asked_for_once(run):
    """A native flush whose workspace is not to be had runs in FP64 tiles and asks again at the next init only."""
    run("""
        h = create(n=130)
        fake.fake_alloc_limit(1 << 20)
        for _ in range(2):
            fake.fake_reset()
            assert init(h) == OK
            for _ in range(9):
                assert propose(h) == OK and accept(h) == OK
            assert sum("k_flush_native" in x for x in names()) == 9 and not any("k_oz_gemm" in x for x in names())
            # the flush's workspace, and the padded elimination's (which runs in its FP64 form)
            assert len(sizes(ok=False)) == 2, sizes(ok=False)
        fake.fake_alloc_limit(1 << 40)
        assert init(h) == OK and propose(h) == OK and accept(h) == OK
        assert "k_flush_native" not in names()[-2] and any("k_oz_gemm" in x for x in names())
    """)


def test_optional_workspaces_come_after_the_required_one(run):
    """A Pfaffian handle that fits beside its elimination slots is initialised, whatever else there is no room for."""
    run("""
        h = create(kind=PF, n=512, W=304)
        slots = 304 * 512 * 512 * 8
        fake.fake_total_limit(sum(sizes()) + slots + (1 << 20))
        assert init(h, PF) == OK
        assert sizes(ok=True)[1:] == [slots]
    """)


@pytest.mark.parametrize("dtype,n,W,padded", [
    ("F64", 55, 1000, False), ("F64", 56, 152, False), ("F64", 56, 153, True), ("F64", 62, 1, False), ("F64", 62, 200, True),
    ("F64", 63, 1, True), ("F64", 64, 1, True), ("F64", 65, 1000, False), ("F64", 72, 304, False), ("F64", 72, 305, True),
    ("F64", 79, 1, False), ("F64", 80, 1, True), ("C128", 56, 1, True), ("C128", 65, 1000, False), ("C128", 72, 1, True)])
def test_inverse_takes_the_faster_form(run, dtype, n, W, padded):
    """Inverses of few small F64 matrices stay with the FP64 form (152 SMs here), those of complex ones do not."""
    run(f"""
        used = lambda: any("k_oz_gemm" in x for x in names())
        h = create(dtype={dtype}, W={W}, n={n}, delay=0)
        fake.fake_reset()
        assert init(h) == OK and used() is {padded}
        grad = lib.lru_slogdet_backward
        grad.argtypes = [C.c_int32, C.c_int64, C.c_int32] + [C.c_void_p] * 6
        fake.fake_reset()
        assert grad({dtype}, {W}, {n}, PTR, PTR, None, None, PTR, None) == OK and used() is {padded}
    """)
