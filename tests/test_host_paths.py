"""The library's host code against a stand-in for the CUDA runtime (fake_cudart.cpp): its own objects,
linked with functions that count launches and can be told to fail, in a process of their own."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

import paper_2511_03683_gb300 as pb

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    b = pb.builder()
    objs = [os.path.join(b.OBJDIR, s + ".o") for s in b.CU_SOURCES + b.CPP_SOURCES]
    newest = max(os.path.getmtime(s) for s in b._sources())
    if not all(os.path.exists(o) and os.path.getmtime(o) >= newest for o in objs):
        b.build(force=True)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))),
                       "include")
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + inc, os.path.join(HERE, "fake_cudart.cpp"),
                           *objs, "-Wl,-Bsymbolic", "-Wl,-z,defs", "-fopenmp", "-o", out])
    return out


PRELUDE = """
import ctypes, sys
import numpy as np
sys.path.insert(0, {root!r})
import synth
import paper_2511_03683_gb300 as pb
pb.LIB_PATH, pb._lib = {lib!r}, None
L = pb.lib()
L.fake_fail.argtypes = L.fake_fail_new.argtypes = [ctypes.c_long]
L.fake_news.restype = L.fake_count.restype = ctypes.c_long

def aligned(n):
    a = np.zeros(n + 256, np.uint8)
    o = -a.ctypes.data % 256
    return a[o:o + n]

def opts(**kw):
    o = pb._DevOpts()
    for k, v in kw.items():
        setattr(o, k, v)
    return o

def device(ch, **kw):
    o, n, h = opts(**kw), ctypes.c_size_t(0), ctypes.c_void_p()
    rc = L.pb_dev_arena_bytes(ch._h, ctypes.byref(o), ctypes.byref(n))
    if rc:
        return rc, None, None
    arena = aligned(n.value)
    rc = L.pb_dev_create(ch._h, ctypes.byref(o), ctypes.c_void_p(arena.ctypes.data), n, None, ctypes.byref(h))
    return rc, h, arena
"""


def child(fake, body):
    src = PRELUDE.format(root=os.path.dirname(HERE), lib=fake) + textwrap.dedent(body)
    r = subprocess.run([sys.executable, "-c", src], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("fail", [False, True])
def test_rk4_eight_step_graph(fake, fail):
    """Every call runs its n steps whatever graphs it replays (one launch for the input, eight per step):
    one by one at first, eight at a time later and in a long call; and where the eight-step graph
    cannot be made, one by one again, with no step done twice or left out and no error."""
    child(fake, f"""
    ch = pb.Channels.from_model(synth.make_window4(8))
    rc, h, arena = device(ch)
    assert rc == pb.PB_OK, L.pb_last_error().decode()
    f = np.zeros(ch.nstate)

    def steps(n):
        a, g = L.fake_count(0), L.fake_count(1)
        rc = L.pb_rtbte_rk4_step(h, ctypes.c_void_p(f.ctypes.data), 1.0, n, None)
        assert rc == pb.PB_OK, L.pb_last_error().decode()
        assert L.fake_count(0) - a == 1 + 8 * n, (n, L.fake_count(0) - a)
        return L.fake_count(1) - g  # graph launches

    assert steps(1) == 1 and steps(9) == 9
    assert steps(41) == 41
    if {fail}:
        L.fake_fail(1)
        assert steps(41) == 41  # the eight-step graph fails: one by one
        assert steps(9) == 9
    else:
        assert steps(41) == 1 + 5  # 1 + 8 * 5
        assert steps(12) == 1 + 1 + 3
        g = np.zeros(ch.nstate)
        f = g  # another vector: the graphs start over, and a long call takes the eight-step one by itself
        assert steps(20) == 20
        assert steps(4001) == 1 + 500
        f = np.zeros(ch.nstate)
        assert steps(4001) == 1 + 500
    L.pb_dev_destroy(h)
    """)


def test_dense_batch_plans_fit_the_arena(fake):
    """pb_batch_arena_bytes bounds the slots of every item size that the autotuner tries and of the
    batch's own, whatever the reach: narrow, ordinary, the whole spectrum, a single energy."""
    child(fake, """
    ms = [synth.make_window4(16, sigma=4e-4), synth.make_window4(17), synth.make_window4(22), synth.make_window4(12, sigma=0.3),
          synth.make_flat_einstein(5), synth.make_tiny(6).with_(T=20.0)]
    chs = [pb.Channels.from_model(m) for m in ms]
    for item in (0, 1024, 3072, 65536):
        for group in [[c] for c in chs] + [chs]:
            arr = (ctypes.c_void_p * len(group))(*[c._h.value for c in group])
            o, n, h = pb._BatchOpts(item, 0, 0, 0), ctypes.c_size_t(0), ctypes.c_void_p()
            assert L.pb_batch_arena_bytes(arr, len(group), ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
            a = aligned(n.value)
            rc = L.pb_batch_create(arr, len(group), ctypes.byref(o), ctypes.c_void_p(a.ctypes.data), n, None, ctypes.byref(h))
            assert rc == pb.PB_OK, L.pb_last_error().decode()
            f = np.zeros(sum(c.nstate for c in group))
            i, c, ms_ = ctypes.c_int32(0), ctypes.c_int32(0), ctypes.c_double(0)
            rc = L.pb_batch_autotune(h, ctypes.c_void_p(f.ctypes.data), None, ctypes.byref(i), ctypes.byref(c), ctypes.byref(ms_))
            assert rc == pb.PB_OK, L.pb_last_error().decode()
            L.pb_batch_destroy(h)
    """)


def test_batch_autotune_times_the_shapes_that_run(fake):
    """Two ring shapes for a float-float batch on the ring (4 x 69 tiles), one for a small list, whose
    kernel has no ring, five for C32: one input launch, then a warm-up and three timed sweeps each."""
    child(fake, """
    def tune(chs, prec):
        arr = (ctypes.c_void_p * len(chs))(*[c._h.value for c in chs])
        o, n, h = pb._BatchOpts(0, 0, prec, 2), ctypes.c_size_t(0), ctypes.c_void_p()
        assert L.pb_batch_arena_bytes(arr, len(chs), ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
        a = aligned(n.value)
        assert L.pb_batch_create(arr, len(chs), ctypes.byref(o), ctypes.c_void_p(a.ctypes.data), n, None, ctypes.byref(h)) == pb.PB_OK
        f = np.zeros(sum(c.nstate for c in chs))
        i, c, ms, before = ctypes.c_int32(0), ctypes.c_int32(0), ctypes.c_double(0), L.fake_count(0)
        assert L.pb_batch_autotune(h, ctypes.c_void_p(f.ctypes.data), None, ctypes.byref(i), ctypes.byref(c), ctypes.byref(ms)) == pb.PB_OK
        got, info = L.fake_count(0) - before, ctypes.c_int32(0)
        assert L.pb_batch_get_info(h, None, None, None, None, ctypes.byref(info)) == pb.PB_OK
        assert info.value == c.value
        L.pb_batch_destroy(h)
        return got, c.value

    small, big = pb.Channels.from_model(synth.make_window4(16)), pb.Channels.from_model(synth.make_window4(24))
    assert tune([small, small], 1) == (1 + 4, 3)
    assert tune([big] * 4, 1)[0] == 1 + 2 * 4
    assert tune([small], 2)[0] == 1 + 5 * 4
    """)


def test_a_failed_batch_plan_leaves_the_one_before_it(fake):
    """The autotuner's plans of the dense FP32 batch: wherever an allocation fails, no copy, clear or launch
    of that plan has been made, so the items on the device still belong to its slots and ranges."""
    child(fake, """
    ch = pb.Channels.from_model(synth.make_window4(16))
    arr = (ctypes.c_void_p * 2)(ch._h.value, ch._h.value)
    o, n = pb._BatchOpts(0, 0, 0, 0), ctypes.c_size_t(0)
    assert L.pb_batch_arena_bytes(arr, 2, ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
    a, f = aligned(n.value), np.zeros(2 * ch.nstate)

    def tune(i):
        h = ctypes.c_void_p()
        assert L.pb_batch_create(arr, 2, ctypes.byref(o), ctypes.c_void_p(a.ctypes.data), n, None, ctypes.byref(h)) == pb.PB_OK
        before = L.fake_count(0) + L.fake_count(3)
        L.fake_fail_new(i)
        rc = L.pb_batch_autotune(h, ctypes.c_void_p(f.ctypes.data), None, None, None, None)
        n_ = L.fake_news()
        L.fake_fail_new(0)
        L.pb_batch_destroy(h)
        if not i:
            global news
            news = n_
        return rc, L.fake_count(0) + L.fake_count(3) - before

    rc, total = tune(0)
    assert rc == pb.PB_OK
    plan, rest = divmod(total - 1 - 3 * 12, 4)  # the input; three sizes' plans and 3 x 4 sweeps; the best's plan
    assert rest == 0 and plan > 10
    whole, failed = {1 + k * (plan + 12) for k in range(4)}, 0
    for i in list(range(1, 40)) + list(range(news // 2, news, news // 60)) + list(range(news - 60, news + 20)):
        rc, done = tune(i)
        if rc != pb.PB_OK:
            assert rc == pb.PB_ENOMEM and done in whole, (i, done, whole)
            failed += 1
    assert failed > 100
    """)


CREATE = {
    "channels": "lambda: build(1)",
    "channels, one callback at a time": "lambda: build(0)",
    "tiles with transport": "lambda: dev(transport=1, adjoint=1)",
    "rows": "lambda: dev(dense_rows=2, transport=1)",
    "dense g32": "lambda: dev(variant=pb.VARIANTS['g32'], adjoint=1)",
    "dense h16, cutoff list": "lambda: dev(cut, variant=pb.VARIANTS['h16'], channel_per_lane=5)",
    "cutoff list, forced tiles": "lambda: dev(cut, dense_rows=3)",
    "paper": "lambda: dev(variant=pb.VARIANTS['paper'])",
    "batch fp32": "lambda: batch(0)",
    "batch ff": "lambda: batch(1)",
    "batch c32": "lambda: batch(2)",
}


@pytest.mark.parametrize("what", list(CREATE))
def test_host_memory_that_runs_out_is_an_error_code(fake, what):
    """The i-th allocation of the call fails, for every i up to the first hundred and then ever larger
    steps: PB_ENOMEM (or success where the failed allocation has a fallback), never an exception through
    the C interface or out of a parallel region."""
    child(fake, f"""
    import os
    m = synth.make_window4(9)
    ch = pb.Channels.from_model(m)
    cut = pb.Channels.from_model(m, g2_min=1e-5, delta_nsigma=6.0)
    rate = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)

    def g2(n, s, p, v, out, user):
        ctypes.memset(out, 0, 8 * n)
        return 0
    g2c = rate(g2)

    def build(threadsafe):
        arrays = [np.ascontiguousarray(a, dtype=np.float64) for a in (m.eps, m.omega, m.win)]
        M = pb._Model()
        M.nk[:] = m.nk
        M.nbands, M.nmodes = m.eps.shape[-1], m.omega.shape[-1]
        M.eps, M.omega, M.win = (a.ctypes.data for a in arrays)
        M.T, M.sigma = m.T, m.sigma
        o = pb._BuildOpts(nthreads=1 if threadsafe else 0, callback_threadsafe=threadsafe, check_closure=1)
        h = ctypes.c_void_p()
        yield lambda: L.pb_build_channels(ctypes.byref(M), ctypes.cast(g2c, ctypes.c_void_p), None, ctypes.byref(o), ctypes.byref(h))
        if h:
            L.pb_channels_free(h)

    def dev(c=ch, **kw):
        o, n, h = opts(**kw), ctypes.c_size_t(0), ctypes.c_void_p()
        assert L.pb_dev_arena_bytes(c._h, ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
        a = aligned(n.value)
        yield lambda: L.pb_dev_arena_bytes(c._h, ctypes.byref(o), ctypes.byref(n)) or L.pb_dev_create(
            c._h, ctypes.byref(o), ctypes.c_void_p(a.ctypes.data), n, None, ctypes.byref(h))
        if h:
            L.pb_dev_destroy(h)

    def batch(prec):
        arr = (ctypes.c_void_p * 2)(ch._h.value, ch._h.value)
        o, n, h = pb._BatchOpts(0, 0, prec, 0), ctypes.c_size_t(0), ctypes.c_void_p()
        f = np.zeros(2 * ch.nstate)
        assert L.pb_batch_arena_bytes(arr, 2, ctypes.byref(o), ctypes.byref(n)) == pb.PB_OK
        a = aligned(n.value)
        yield lambda: L.pb_batch_arena_bytes(arr, 2, ctypes.byref(o), ctypes.byref(n)) or L.pb_batch_create(
            arr, 2, ctypes.byref(o), ctypes.c_void_p(a.ctypes.data), n, None, ctypes.byref(h)) or L.pb_batch_autotune(
            h, ctypes.c_void_p(f.ctypes.data), None, None, None, None)
        if h:
            L.pb_batch_destroy(h)

    i, failed = 0, 0
    while True:
        i += 1 + max(0, i - 100) // 20
        it = ({CREATE[what]})()
        call = next(it)
        L.fake_fail_new(i)
        rc = call()
        done = L.fake_news() < i
        L.fake_fail_new(0)
        assert rc in (pb.PB_OK, pb.PB_ENOMEM), (i, rc, L.pb_last_error().decode())
        failed += rc == pb.PB_ENOMEM
        next(it, None)
        if done:
            assert rc == pb.PB_OK
            break
    assert failed >= 3, failed
    """)
