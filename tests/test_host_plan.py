"""The plan's host code (ef_plan.cpp) on the CPU, against a CUDA runtime that records instead of running
(fake_cuda.cpp): which shape, parts and workspaces a call uses, and what it waits for."""
import ctypes
import os
import subprocess

import pytest

import paper_1704_07369_gb300 as ef

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1704_07369_gb300", "csrc")

FIELDS = ("kind", "stream", "event", "N", "ncells", "cells_off", "nsplit", "cluster", "threads", "occ", "sg_global",
          "clusters", "fh", "sg", "part", "fin", "paired", "prefetch")


class _Rec(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int64) for n in FIELDS]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfakeplan.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + os.path.join(cuda, "include"),
                    "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, os.path.join(HERE, "fake_cuda.cpp"),
                    os.path.join(CSRC, "ef_plan.cpp"), "-o", out, "-lpthread", "-Wl,-Bsymbolic"], check=True)      # its own runtime, whatever else is loaded
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = ctypes.c_int64
    lib.fake_used.restype = ctypes.c_size_t
    lib.fake_peak.restype = ctypes.c_size_t
    lib.ef_last_error.restype = ctypes.c_char_p
    return lib


@pytest.fixture(autouse=True)
def _plain_environment(monkeypatch):
    for v in ("EF_SHAPE", "EF_AUTOTUNE", "EF_AUTOTUNE_CACHE", "EF_AUTOTUNE_LOG", "EF_CONCURRENT_CLASSES"):
        monkeypatch.delenv(v, raising=False)


class Plan:
    """A plan of the host code, its calls returning what they enqueued."""

    def __init__(self, lib, d, N, kernel, R, prec, cells=None):
        self.lib, self.cells = lib, cells
        self.h = ctypes.c_void_p()
        if cells is None:
            st = lib.ef_plan_create(d, N, ctypes.c_double(8.0), kernel, R, prec, ctypes.byref(self.h))
        else:
            Ns = (ctypes.c_int * len(cells))(*cells)
            st = lib.ef_plan_create_batched(d, ctypes.c_int64(len(cells)), Ns, ctypes.c_double(8.0), kernel, R, prec,
                                            ctypes.byref(self.h))
        assert st == ef.EF_OK, lib.ef_last_error()
        lib.fake_clear()

    def _log(self):
        buf = (_Rec * 4096)()
        n = self.lib.fake_log(buf, ctypes.c_int64(4096))
        assert n <= 4096
        self.lib.fake_clear()
        return list(buf[:n])

    def collide(self, n, stream=0x10):
        st = self.lib.ef_collide(self.h, ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 21), ctypes.c_int64(n),
                                 ctypes.c_void_p(stream))
        assert st == ef.EF_OK, self.lib.ef_last_error()
        return self._log()

    def close(self):
        self.lib.ef_plan_destroy(self.h)


def launches(log):
    return [r for r in log if r.kind == 0]


def finishes(log):
    return [r for r in log if r.kind == 1]


F32, F64, MAXWELL, HARD = ef.EF_PREC_F32, ef.EF_PREC_F64, ef.EF_KERNEL_MAXWELL, ef.EF_KERNEL_HARD_SPHERE
# d, N, kernel, R, precision: plans whose kernels keep the forward spectrum in a workspace (N = 64 FP64: the
# accumulators too)
SPECTRUM = [(3, 16, HARD, 16, F64), (3, 64, HARD, 16, F64), (2, 24, MAXWELL, 16, F64), (2, 16, MAXWELL, 16, F32),
            (3, 12, HARD, 16, F32)]


def workspaces(log):
    """Every workspace address the launches of a call were given."""
    out = set()
    for r in log:
        if r.kind in (0, 1):
            out |= {("fh", r.fh), ("sg", r.sg), ("part", r.part), ("fin", r.fin)}
    return {x for x in out if x[1]}


@pytest.mark.parametrize("d,N,kernel,R,prec", SPECTRUM)
@pytest.mark.parametrize("n", [1, 3, 20000])
def test_graphs_and_calls_have_workspaces_of_their_own(lib, d, N, kernel, R, prec, n):
    p = Plan(lib, d, N, kernel, R, prec)
    seen = [workspaces(p.collide(n))]
    if n == 1 and N != 12:               # cells of 1728 points: a split would cost more than it gives
        assert launches(p.collide(n))[0].nsplit > 1
    if n == 20000:
        assert launches(p.collide(n))[0].nsplit == 1
    for g in range(4):
        stream = 0x100 + 16 * g
        lib.fake_begin_capture(ctypes.c_void_p(stream), ctypes.c_ulonglong(g + 1))
        log = p.collide(n, stream)
        again = p.collide(n, stream)
        lib.fake_end_capture(ctypes.c_void_p(stream))
        assert workspaces(again) == workspaces(log)          # one stream of one capture: in order
        assert not [r for r in log if r.kind in (2, 3)]
        seen.append(workspaces(log))
    for i in range(5):
        assert seen[i]
        for j in range(i):
            assert not seen[i] & seen[j], (i, j)
    # a graph that is gone gives its workspace back
    lib.fake_destroy_graph(ctypes.c_ulonglong(2))
    lib.fake_begin_capture(ctypes.c_void_p(0x500), ctypes.c_ulonglong(9))
    assert workspaces(p.collide(n, 0x500)) == seen[2]
    lib.fake_end_capture(ctypes.c_void_p(0x500))
    for g in (1, 3, 4, 9):
        lib.fake_destroy_graph(ctypes.c_ulonglong(g))
    p.close()


@pytest.mark.parametrize("d,N,kernel,R,prec", SPECTRUM)
@pytest.mark.parametrize("first,second", [(1, 1), (20000, 20000), (1, 20000), (20000, 1)])
def test_calls_of_two_streams_wait_for_each_other(lib, d, N, kernel, R, prec, first, second):
    p = Plan(lib, d, N, kernel, R, prec)
    a = p.collide(first, 0x10)
    b = p.collide(second, 0x20)
    assert a[-1].kind == 2 and a[-1].stream == 0x10
    assert b[0].kind == 3 and b[0].stream == 0x20 and b[0].event == a[-1].event
    p.close()


def test_register_kernels_unsplit_need_no_order(lib):
    """Their launches share nothing between calls: streams stay independent."""
    p = Plan(lib, 3, 32, HARD, 16, F32)
    for stream in (0x10, 0x20):
        log = p.collide(5000, stream)
        assert [r.kind for r in log] == [0] and log[0].nsplit == 1 and not workspaces(log)
    p.close()


@pytest.mark.parametrize("prec", [F32, F64])
def test_rk3_calls_wait_for_each_other(lib, prec):
    """The stage buffers are the plan's."""
    p = Plan(lib, 3, 32, HARD, 16, prec)
    n = 600
    assert lib.ef_plan_reserve(p.h, ctypes.c_int64(n)) == ef.EF_OK
    logs = []
    for stream in (0x10, 0x20):
        assert lib.ef_rk3_step(p.h, ctypes.c_void_p(1 << 20), ctypes.c_double(0.01), 1, None, ctypes.c_int64(n),
                               ctypes.c_void_p(stream)) == ef.EF_OK
        logs.append(p._log())
    assert logs[0][-1].kind == 2 and logs[1][0].kind == 3 and logs[1][0].event == logs[0][-1].event
    p.close()


def call_info(p, n, split):
    out = (ctypes.c_int64 * 8)()
    assert p.lib.ef_plan_call_info(p.h, 0, ctypes.c_int64(n), split, out) == ef.EF_OK
    return dict(zip(("parts", "cluster", "threads", "variant", "launches", "clusters"), out))


@pytest.mark.parametrize("d,N,kernel,R,prec", SPECTRUM + [(3, 32, MAXWELL, 32, F32), (3, 48, HARD, 32, F32), (3, 32, MAXWELL, 32, F64)])
@pytest.mark.parametrize("n", [1, 2, 7])
def test_a_capture_without_a_workspace_launches_whole_cells(lib, d, N, kernel, R, prec, n):
    """Four captures get workspaces; the fifth launches what ef_plan_call_info gives for a call that may not be
    split."""
    p = Plan(lib, d, N, kernel, R, prec)
    split, whole = call_info(p, n, 1), call_info(p, n, 0)
    assert whole["parts"] == 1 and whole["launches"] == 1
    for g in range(5):
        stream = 0x100 + 16 * g
        lib.fake_begin_capture(ctypes.c_void_p(stream), ctypes.c_ulonglong(g + 1))
        r = launches(p.collide(n, stream))[0]
        lib.fake_end_capture(ctypes.c_void_p(stream))
        want = split if g < 4 else whole
        assert (r.nsplit, r.cluster, r.threads, r.occ) == (want["parts"], want["cluster"], want["threads"], want["variant"])
    for g in range(5):
        lib.fake_destroy_graph(ctypes.c_ulonglong(g + 1))
    p.close()


@pytest.mark.parametrize("d,N,kernel,R,prec,n", [(3, 16, HARD, 16, F64, 2), (3, 16, HARD, 16, F64, 4), (2, 64, MAXWELL, 16, F64, 2)])
def test_whole_cells_do_not_take_the_shape_chosen_for_parts(lib, d, N, kernel, R, prec, n):
    """Here parts run best one line transform a team on many small CTAs; a whole cell, whose every pass ends in
    a cluster barrier, on fewer."""
    p = Plan(lib, d, N, kernel, R, prec)
    split, whole = call_info(p, n, 1), call_info(p, n, 0)
    assert split["parts"] > 1 and whole["parts"] == 1
    assert whole["cluster"] < split["cluster"]
    p.close()


@pytest.mark.parametrize("n,split", [(400, True), (2400, True), (3000, False), (6000, False), (200000, False)])
def test_ragged_plans_split_only_what_is_resident_at_once(lib, n, split):
    """Every part of a split launch has a cluster of its own, whatever smaller count the tuner timed: small cells
    are resident by the thousand, and parts of more would be rounds of repeated work and workspaces that grow
    with the batch."""
    p = Plan(lib, 2, None, MAXWELL, 16, F32, cells=[8] * n)
    used = lib.fake_used()
    r = launches(p.collide(n))[0]
    assert (r.nsplit > 1) == split
    assert r.clusters >= n * r.nsplit or r.nsplit == 1
    assert used <= (64 << 20) + 64 * n
    p.close()


@pytest.mark.parametrize("d,N,kernel,R,prec,cells", [(3, 32, MAXWELL, 32, F32, None), (3, 32, HARD, 32, F64, None), (2, 64, MAXWELL, 16, F64, None),
                                                     (3, 64, HARD, 16, F64, None), (3, None, HARD, 32, F32, [32] * 20 + [48] * 3)])
def test_a_plan_without_room_for_parts_and_captures_still_works(lib, d, N, kernel, R, prec, cells):
    """The workspaces of split launches and of captures are dropped before a plan is refused: down to what whole
    cells need, every limit of device memory below the full plan's is enough, and nothing is left behind."""
    n = 1 if cells is None else len(cells)
    base = lib.fake_used()
    lib.fake_peak()
    p = Plan(lib, d, N, kernel, R, prec, cells)
    full = lib.fake_peak() - base
    assert any(r.nsplit > 1 for r in launches(p.collide(n)))
    p.close()
    assert lib.fake_used() == base
    kinds = set()
    frac = 1.0
    try:
        while True:
            frac *= 0.75
            lib.fake_limit(ctypes.c_size_t(base + int(full * frac)))
            try:
                p = Plan(lib, d, N, kernel, R, prec, cells)
            except AssertionError:
                break
            assert lib.cudaPeekAtLastError() == 0
            log = p.collide(n)
            kinds.add(any(r.nsplit > 1 for r in launches(log)))
            lib.fake_begin_capture(ctypes.c_void_p(0x100), ctypes.c_ulonglong(1))
            captured = p.collide(n, 0x100)
            lib.fake_end_capture(ctypes.c_void_p(0x100))
            assert len(launches(captured)) == len(launches(log))
            lib.fake_destroy_graph(ctypes.c_ulonglong(1))
            p.close()
            assert lib.fake_used() == base
    finally:
        lib.fake_limit(ctypes.c_size_t(1 << 40))
    assert lib.fake_used() == base
    assert kinds == {True, False}
    assert frac <= 0.35


@pytest.mark.parametrize("d,N,R,prec,kernel", [(3, 24, 16, F64, HARD), (2, 32, 16, F64, MAXWELL), (3, 24, 16, F32, HARD), (2, 16, 16, F32, MAXWELL)])
def test_the_tuner_times_nothing_twice(lib, d, N, R, prec, kernel):
    """Four launches of each candidate: whole cells, in FP32 with and without the prefetch, and parts with the
    better of the two (the FP64 kernel has no prefetch)."""
    h = ctypes.c_void_p()
    cells = [N] * 20
    lib.fake_clear()
    assert lib.ef_plan_create_batched(d, ctypes.c_int64(20), (ctypes.c_int * 20)(*cells), ctypes.c_double(8.0), kernel, R, prec,
                                      ctypes.byref(h)) == ef.EF_OK
    buf = (_Rec * 8192)()
    n = lib.fake_log(buf, ctypes.c_int64(8192))
    lib.fake_clear()
    assert n <= 8192
    timed = {}
    for r in launches(buf[:n]):
        shape = (r.cluster, r.threads, r.occ, r.sg_global, r.paired)
        timed.setdefault(shape, {}).setdefault((r.nsplit, r.prefetch), 0)
        timed[shape][(r.nsplit, r.prefetch)] += 1
    assert timed
    for shape, forms in timed.items():
        assert set(forms.values()) == {4}
        whole = [f for f in forms if f[0] == 1]
        assert len(whole) == (1 if prec == F64 else 2)
        assert len(forms) - len(whole) <= 1
    lib.ef_plan_destroy(h)
