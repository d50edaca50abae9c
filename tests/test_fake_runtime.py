"""Host side of the library against a CUDA runtime without a device (fake_cudart.c), so that what needs a second
GPU, a failing call or a capture in progress is looked at on the CPU.  Each test is a child process with the
runtime preloaded."""
import os
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = r"""
import ctypes as C, sys
F = C.CDLL(sys.argv[1]); D = C.CDLL(sys.argv[2])
F.fake_log.restype = C.c_char_p
vp = C.c_void_p
class Cfg(C.Structure):
    _fields_ = [("n_layers", C.c_int), ("dims", C.POINTER(C.c_int)), ("w_bits", C.c_int), ("a_bits", C.c_int), ("omega0", C.c_float),
                ("w_gran", C.c_int), ("a_gran", C.c_int), ("rotation", C.c_int), ("activation", C.c_int), ("act_s0", C.c_float)]
D.dhq_forward.argtypes = [vp, vp, C.c_int64, vp, vp]; D.dhq_calibrate.argtypes = [vp, vp, C.c_int64, vp]
D.dhq_destroy.argtypes = [vp]; D.dhq_destroy.restype = None; D.dhq_release_cached_memory.restype = None
mem = (C.c_float * 4096)()                      # stands for every buffer of the caller
ptr = C.addressof(mem)
def prepare(width=64, w_bits=8, a_bits=8, w_gran=0, a_gran=0, rotation=0, expect=0):
    dims = (C.c_int * 5)(2, width, width, width, 3)
    cfg = Cfg(4, dims, w_bits, a_bits, 30.0, w_gran, a_gran, rotation, 0, 0.0)
    W = (vp * 4)(*[ptr] * 4); h = vp()
    rc = D.dhq_prepare(C.byref(cfg), W, W, None, C.byref(h))
    assert rc == expect, rc
    return h
def forward(h, stream=0, n=100, expect=0):
    rc = D.dhq_forward(h, ptr, n, ptr, stream)
    assert rc == expect, rc
def calibrate(h, stream=0, n=100, expect=0):
    rc = D.dhq_calibrate(h, ptr, n, stream)
    assert rc == expect, rc
def log():
    lines = F.fake_log().decode().split(); F.fake_clear()
    return [(w, int(d), int(a)) for w, d, a in (x.split(":") for x in lines)]
def set_(what, v): F.fake_set(what.encode(), v)
def early(): return [a for w, _, a in log() if w == "forward"][-1]
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2508_13478_b200 import build
    lib = build.build()
    fake = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", fake, os.path.join(HERE, "fake_cudart.c")], check=True)

    def child(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body), fake, lib], capture_output=True, text=True,
                           timeout=120, env=dict(os.environ, LD_PRELOAD=fake))
        assert r.returncode == 0, r.stdout + r.stderr
    return child


def test_destroy_waits_for_the_handles_device(run):
    run("""
    h = prepare(); log()
    F.cudaSetDevice(1); log()
    D.dhq_destroy(h)
    got = log()
    assert ("sync", 0, 0) in got and not any(w == "sync" and d == 1 for w, d, _ in got), got
    assert got[-1] == ("set_device", 1, 1), got           # the caller's device is current again
    F.cudaSetDevice(0); log()
    h = prepare()
    assert not any(w == "malloc" for w, _, _ in log())     # the block of the first handle
    set_("fail_sync", 1); log()
    D.dhq_destroy(h)                                       # could not wait: the block is not kept
    assert any(w == "free" for w, _, _ in log())
    set_("fail_sync", 0)
    prepare()
    assert any(w == "malloc" for w, _, _ in log())
    """)


@pytest.mark.parametrize("kw", ["", "width=512, w_gran=1, a_gran=1", "width=128, w_gran=1, a_gran=1, rotation=1"])
def test_only_a_launch_behind_an_ordinary_one_in_its_stream_is_early(run, kw):
    run(f"""
    h = prepare({kw})
    calibrate(h, 16); forward(h, 16); assert early() == 0
    forward(h, 16); assert early() == 1
    forward(h, 32); assert early() == 0                    # another stream: not behind those
    forward(h, 32); assert early() == 1
    forward(h, 16); assert early() == 0
    if {"a_gran=1" not in kw}:
        calibrate(h, 16); set_("capturing", 1); forward(h, 48); assert early() == 0   # only recorded
        set_("capturing", 0); forward(h, 48); assert early() == 0
        calibrate(h, 16); set_("fail_launch", 1); forward(h, 16, expect=4)             # enqueued nothing
        set_("fail_launch", 0); forward(h, 16); assert early() == 0
    """)


def test_device_memory_is_cleared_before_a_handle_uses_it(run):
    run("""
    for kw in (dict(), dict(width=512, a_gran=1), dict(width=128, w_gran=1, a_gran=1, rotation=1)):
        D.dhq_release_cached_memory(); log()
        prepare(**kw)
        got = log()
        blocks, cleared = [a for w, _, a in got if w == "malloc"], [a for w, _, a in got if w == "memset"]
        assert cleared[0] == blocks[0] and len(cleared) == len(blocks), got
    """)


def test_a_calibration_that_cannot_allocate_leaves_the_scales(run):
    run("""
    h = prepare(width=128, w_gran=1, rotation=1)           # calibrates layer by layer, through scratch memory
    D.dhq_get_act_absmax.argtypes = [vp, C.c_int, C.POINTER(C.c_float), vp]
    D.dhq_set_act_absmax.argtypes = [vp, C.c_int, C.c_float, vp]
    for l in range(1, 5):
        assert D.dhq_set_act_absmax(h, l, 3.0, None) == 0
    set_("fail_malloc", 1); calibrate(h, 16, expect=3); set_("fail_malloc", 0)
    a = C.c_float()
    for l in range(1, 5):
        assert D.dhq_get_act_absmax(h, l, C.byref(a), None) == 0 and a.value == 3.0, (l, a.value)
    """)


def test_releasing_cached_memory_forgets_what_a_device_was_told(run):
    # a program that resets the device starts from nothing: no kept block, no kernel attribute taken for granted
    run("""
    h = prepare(); first = [w for w, _, _ in log()].count("attribute")
    assert first > 0
    D.dhq_destroy(h); prepare(); assert "attribute" not in [w for w, _, _ in log()]
    D.dhq_release_cached_memory(); log()
    prepare()
    names = [w for w, _, _ in log()]
    assert names.count("attribute") == first and "malloc" in names, names
    """)
