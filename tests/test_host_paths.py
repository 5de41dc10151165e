"""The library's host side on a fake CUDA runtime (fake_cudart.cpp: device memory is
host memory, kernels do not run), for what a GPU run cannot show safely: failed
allocations, buffers of another GPU, and work that a call leaves on the legacy stream,
which a non-blocking stream does not wait for.  Each test runs its body in a child
process with the fake preloaded."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2507_00528_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = r"""
import ctypes as C, struct, sys
sys.path.insert(0, {root!r})
from paper_2507_00528_gb300 import _lib
L = _lib.load()
fake = C.CDLL(None)
for f in ("fake_plant", "fake_foreign", "fake_copies", "cudaMalloc"):
    getattr(fake, f).argtypes = dict(fake_plant=[C.c_size_t, C.c_char_p], cudaMalloc=[C.c_void_p, C.c_size_t]).get(
        f, [C.c_void_p])
INVALID, OOM, CUDA = -1, -2, -3
ST = C.c_void_p(0x1234)  # a stream that is not the legacy one

def device(values, fmt):
    # a device array of the values
    raw = struct.pack("%d%s" % (len(values), fmt), *values)
    p = C.c_void_p()
    assert fake.cudaMalloc(C.byref(p), len(raw)) == 0
    C.memmove(p, raw, len(raw))
    return p.value

def found(radial=40, angular=10, most=10, flags=16, err=0):
    # what a build's search reports to the host next (BuildResult)
    fake.fake_plant(32, struct.pack("qqiiii", radial, angular, most, flags, err, 0))

def batch():
    return _lib.Batch(1, 2, device([0, 2], "i"), device([1.0] * 6, "d"), device([0, 1], "i"),
                      device([9.0, 0, 0, 0, 9.0, 0, 0, 0, 9.0], "d"))

def model():
    m = C.c_void_p()
    assert L.gnep_create(C.byref(m), 2, None, 7.0, 4.0, 4, 4, 8, 8, 4, 0, 30, 0, 0) == 0
    return m

def built(m, b):
    nl = C.c_void_p()
    found()
    assert L.gnep_build_neighbors(m, C.byref(b), C.byref(nl), ST) == 0, L.gnep_last_error()
    return nl

def labels():
    return _lib.Labels(device([0.0], "d"), device([0.0] * 6, "f"), device([0.0] * 6, "d"), 1.0, 1.0, 0.1, 0.0, 0)
"""


@pytest.fixture(scope="session")
def fake(tmp_path_factory):
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", so], check=True)
    return so


@pytest.fixture
def run(fake):
    def run(body):
        code = PRELUDE.format(root=os.path.dirname(HERE)) + textwrap.dedent(body)
        p = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LD_PRELOAD=fake), capture_output=True,
                           text=True, timeout=120)
        assert p.returncode == 0, p.stderr[-3000:]
    return run


def test_nothing_is_left_on_the_legacy_stream(run, tmp_path):
    """Every call leaves its device work on its own stream, or has waited for it."""
    run(f"""
    m = model()
    assert fake.fake_legacy_pending() == 0
    b = batch()
    nl = built(m, b)
    assert fake.fake_legacy_pending() == 0
    found(radial=4000, angular=1000)  # the lists and the workspace grow
    before = fake.fake_memsets_on_streams()
    assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == 0
    assert fake.fake_legacy_pending() == 0 and fake.fake_memsets_on_streams() >= before + 2
    found(err=4)  # an asymmetric list, seen by the next molecular dynamics step
    v = [device([0.0] * 6, "d") for _ in range(2)]
    im, F = device([1.0, 1.0], "d"), device([0.0] * 6, "f")
    assert L.gnep_md_verlet(m, nl, v[0], v[1], im, F, 1.0, None, ST) == INVALID
    assert fake.fake_legacy_pending() == 0
    fake.fake_plant(4, struct.pack("i", 1))  # a loss that was not finite
    assert L.gnep_sync_status(m, ST) == -5
    assert fake.fake_legacy_pending() == 0
    fake.fake_plant(4, None)
    path = {str(tmp_path / "m.ckpt")!r}.encode()
    assert L.gnep_save(m, path) == 0 and L.gnep_load(m, path) == 0
    assert fake.fake_legacy_pending() == 0
    """)


def test_a_list_whose_rebuild_failed_is_refused_until_it_is_rebuilt(run):
    """Each allocation of a rebuild that grows the lists fails in turn.  The first, the
    scratch, comes before any change; after the others no call may use the arrays, and
    the next rebuild groups the species again."""
    run("""
    m, b, y = model(), batch(), labels()
    nl = built(m, b)
    found(radial=4000, angular=1000)
    fake.fake_fail_alloc(0)
    assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == 0
    total = fake.fake_allocs()
    assert total >= 12  # scratch, 3 + 5 pair arrays, 2 for the grouping, the workspace
    F = device([0.0] * 6, "f")
    pos, vel, im = device([1.0] * 6, "d"), device([0.0] * 6, "d"), device([1.0, 1.0], "d")
    off = (C.c_int32 * 3)()
    g = C.c_void_p()
    sched = (1e-3, 1e-6, 10, 100, 0.9, 0.999, 1e-8, 0.0)
    def calls(nl):
        return [L.gnep_forward(m, nl, None, None, F, None, ST), L.gnep_loss(m, nl, C.byref(y), None, ST),
                L.gnep_loss_grad(m, nl, C.byref(y), None, None, ST), L.gnep_descriptors(m, nl, None, ST),
                L.gnep_descriptors_noalloc(m, nl, device([0.0] * 50, "f"), ST),
                L.gnep_nlist_export(nl, 0, off, None, None, ST),
                L.gnep_compute_descriptor_scale(m, nl, ST),
                L.gnep_graph_create(m, nl, C.byref(y), None, *(C.c_double(x) if isinstance(x, float) else x
                                                               for x in sched), ST, C.byref(g))]
    for nth in range(1, total + 1):
        nl = built(m, b)
        found(radial=4000, angular=1000)
        fake.fake_fail_alloc(nth)
        assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == OOM, nth
        fake.fake_fail_alloc(0)
        n = fake.fake_launches()
        if nth == 1:
            assert calls(nl) == [0] * 8
        else:
            assert calls(nl) == [INVALID] * 8, nth
            assert L.gnep_md_verlet(m, nl, pos, vel, im, F, 1.0, None, ST) == INVALID
            assert fake.fake_launches() == n  # nothing ran on the broken list
        fake.fake_fail_alloc(0)
        found(radial=4000, angular=1000, flags=0)  # the same species as the failed batch
        n = fake.fake_launches()
        assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == 0
        regrouped = fake.fake_launches() - n
        n = fake.fake_launches()
        assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == 0
        assert regrouped - (fake.fake_launches() - n) == (0 if nth == 1 else 3), nth
        assert calls(nl) == [0] * 8
        assert L.gnep_md_verlet(m, nl, pos, vel, im, F, 1.0, None, ST) == 0
        L.gnep_nlist_destroy(nl)
    """)


def test_a_refused_batch_leaves_captured_graphs(run):
    """Each refusal of a rebuild leaves the list as it was, so that graphs captured on it
    still launch; a rebuild that went through, or a molecular dynamics step that moved the
    list's positions, ends them."""
    run("""
    m, b, y = model(), batch(), labels()
    nl = built(m, b)
    def graph():
        g = C.c_void_p()
        assert L.gnep_graph_create(m, nl, C.byref(y), None, 1e-3, 1e-6, 10, 100, 0.9, 0.999, 1e-8, 0.0, ST,
                                   C.byref(g)) == 0
        return g
    g = graph()
    for seen, rc in ((dict(flags=1), INVALID), (dict(flags=2), INVALID), (dict(flags=4), INVALID),
                     (dict(flags=8), INVALID), (dict(radial=1 << 31), -4), (dict(angular=1 << 31), -4)):
        found(**seen)
        assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == rc, seen
        assert L.gnep_graph_launch(g, ST) == 0, seen
    found()
    assert L.gnep_rebuild_neighbors(m, C.byref(b), nl, ST) == 0
    assert L.gnep_graph_launch(g, ST) == INVALID
    g = graph()
    found(flags=8)  # positions that are not numbers after the drift
    F = device([0.0] * 6, "f")
    pos, vel, im = device([1.0] * 6, "d"), device([0.0] * 6, "d"), device([1.0, 1.0], "d")
    assert L.gnep_md_verlet(m, nl, pos, vel, im, F, 1.0, None, ST) == INVALID
    assert L.gnep_graph_launch(g, ST) == INVALID
    """)


def test_buffers_that_kernels_must_not_touch_are_copied(run):
    """Batch arrays and outputs in this GPU's memory are used in place; in another GPU's,
    or off their type's alignment, they are copied."""
    run("""
    m, b = model(), batch()
    nl = built(m, b)
    names = ("struct_off", "pos", "type", "cell")
    assert [fake.fake_copies(getattr(b, f)) for f in names] == [0] * 4
    for f in names:
        other = batch()
        fake.fake_foreign(getattr(other, f))
        found()
        assert L.gnep_rebuild_neighbors(m, C.byref(other), nl, ST) == 0
        assert fake.fake_copies(getattr(other, f)) == 1, f
    for f, values, fmt in (("pos", [1.0] * 6, "d"), ("cell", [9.0] * 9, "d"), ("type", [0, 1], "i")):
        other, room = batch(), device([0] * 100, "b")
        at = room + (4 if fmt == "d" else 2)
        C.memmove(at, struct.pack("%d%s" % (len(values), fmt), *values), 4 * len(values))
        setattr(other, f, at)
        found()
        assert L.gnep_rebuild_neighbors(m, C.byref(other), nl, ST) == 0
        assert fake.fake_copies(at) == 1, f
    sizes = (("f", 2), ("d", 1), ("f", 6), ("d", 6))
    for k in range(4):
        for foreign, shift in ((False, 0), (True, 0), (False, 2)):
            out = [device([0.0] * (n + 1), t) for t, n in sizes]
            out[k] += shift
            if foreign:
                fake.fake_foreign(out[k])
            assert L.gnep_forward(m, nl, *out, ST) == 0
            assert [fake.fake_copies(p) for p in out] == [int(q == k and (foreign or shift > 0)) for q in range(4)]
    F = device([0.0] * 6, "f")
    pos, vel, im, E = device([1.0] * 6, "d"), device([0.0] * 6, "d"), device([1.0, 1.0], "d"), device([0.0], "d")
    for copies in (0, 1):
        found()
        assert L.gnep_md_verlet(m, nl, pos, vel, im, F, 1.0, E, ST) == 0
        assert fake.fake_copies(E) == copies
        fake.fake_foreign(E)
    """)
