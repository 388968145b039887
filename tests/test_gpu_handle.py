"""GPU tests of what a mesh handle keeps between calls: recorded graphs and
their constants, steady weights, T^0, options, the tuner, device memory."""
import ctypes

import numpy as np
import pytest

import paper_2104_09189_gb300 as sl
import sl_inputs as si
from gpu_helpers import DeviceRun

pytestmark = pytest.mark.gpu

PRECISIONS = pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])


class Batch:
    """Several meshes on one handle, with their values."""

    def __init__(self, sizes, precision=sl.SL_FP64):
        import torch
        self.meshes = [si.grid_mesh(M, 0.25, M) for M in sizes]
        self.h = sl.sl_mesh_create(*sl.pack_meshes([(m.xy, m.tri) for m in self.meshes]), precision=precision)
        self.v0 = torch.tensor(np.concatenate([si.gaussian(m.xy) for m in self.meshes]), device="cuda",
                               dtype=torch.float64 if precision == sl.SL_FP64 else torch.float32)

    def __del__(self):
        sl.sl_mesh_destroy(self.h)


def status_of(call, *args, **kw):
    try:
        call(*args, **kw)
        return sl.SL_OK
    except sl.SLError as e:
        return e.status


def t0_of(h, n):
    import torch
    j = torch.empty(n, dtype=torch.int32, device="cuda")
    sl.sl_mesh_get_t0(h, j)
    return j


def run_from_start(h, probs, v0, chunks, use_graph):
    """(V, T0, status) after runs of the given numbers of steps from the initial T0."""
    import torch
    v, w = v0.clone(), torch.empty_like(v0)
    sl.sl_mesh_reset_t0(h)
    n, status = 0, sl.SL_OK
    for c in chunks:
        status = max(status, status_of(sl.sl_run, h, probs, n, c, v, w, use_graph=use_graph))
        n += c
    return v, t0_of(h, v.numel()), status


def fields_of(kinds):
    make = {"rotation": si.rotation_field, "swirl": si.swirl_field, "zero": si.zero_field,
            "slow": lambda: si.rotation_field(1.0)}
    return sl.problems([(f.kind, 0.04, f.packed()) for f in (make[k]() for k in kinds)])


@pytest.mark.parametrize("kernel", [2, 1], ids=["fast", "plain"])
@pytest.mark.parametrize("eager_steps", [6, 40])
def test_a_launched_run_between_replays_of_a_batch(eager_steps, kernel):
    """A batch's recorded graph reads its constants from a buffer of the handle,
    which a run that is launched step by step rewrites, and replaces where it
    needs more of it."""
    b = Batch((20, 33, 9))
    sl.sl_mesh_set_option(b.h, sl.SL_OPT_KERNEL, kernel)
    A, B = fields_of(("rotation", "swirl", "zero")), fields_of(("swirl", "slow", "rotation"))
    want = run_from_start(b.h, A, b.v0, (6,), False)
    v, w = b.v0.clone(), b.v0.clone()
    for use in ("launched", "recorded", "replayed", "after the other run"):
        if use == "after the other run":
            v.copy_(b.v0)
            sl.sl_run(b.h, B, 0, eager_steps, v, w, use_graph=False)
        v.copy_(b.v0)
        sl.sl_mesh_reset_t0(b.h)
        sl.sl_run(b.h, A, 0, 6, v, w, use_graph=True)
        assert bool((v == want[0]).all()) and bool((t0_of(b.h, v.numel()) == want[1]).all()), use


@pytest.mark.parametrize("problems", [1, 3])
@pytest.mark.parametrize("call", ["step", "run"])
def test_a_capturing_stream_is_refused(call, problems):
    """A caller's graph would keep addresses of the handle's constants, which
    later calls rewrite or free, and its tables, which follow the field."""
    import torch
    b = Batch((20, 33, 9)[:problems])
    probs = fields_of(("rotation",) * problems)
    w = torch.empty_like(b.v0)
    if call == "run":
        sl.sl_mesh_set_option(b.h, sl.SL_OPT_ASYNC, 1)
    sl.sl_step(b.h, probs, 0, b.v0, w)                 # everything a step allocates
    torch.cuda.synchronize()
    with torch.cuda.graph(torch.cuda.CUDAGraph(), capture_error_mode="thread_local"):
        if call == "step":
            got = status_of(sl.sl_step, b.h, probs, 1, b.v0, w)
        else:
            got = status_of(sl.sl_run, b.h, probs, 1, 2, b.v0, w, use_graph=False, stats=False)
    assert got == sl.SL_E_CUDA
    sl.sl_step(b.h, probs, 1, b.v0, w)                 # the handle goes on
    sl.sl_mesh_status(b.h)


@pytest.mark.parametrize("precision,records,split", [(sl.SL_FP64, 0, 0), (sl.SL_FP64, 1, 0), (sl.SL_FP64, 0, 1),
                                                     (sl.SL_FP32, 0, 0)],
                         ids=["fp64", "fp64-records8", "fp64-split", "fp32"])
def test_every_hop_cap_where_the_field_vanishes(precision, records, split):
    """The swirl's feet are their nodes at t = 1/2, cells away from the triangles
    of the step before: the walk back there keeps to a cap of the caller's, the
    same with and without the counting variant."""
    m = si.grid_mesh(60, 0.25, 7)
    g = DeviceRun(m, si.swirl_field(), 0.05, precision=precision)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_RECORDS, records)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_SPLIT, split)
    t = g.torch
    v = g.to_dev(si.cosine_bump(m.xy))
    w = t.empty_like(v)
    sl.sl_step(g.h, g.probs, 1, v, w)
    start = t0_of(g.h, m.n_nodes)
    outcomes = set()
    for cap in range(1, 13):
        sl.sl_mesh_set_option(g.h, sl.SL_OPT_WALK_CAP, cap)
        got = []
        for debug in (True, False):
            sl.sl_mesh_set_t0(g.h, start)
            w = t.empty_like(v)
            moves = t.zeros(m.n_nodes, dtype=t.int32, device=g.dev)
            sl.sl_step(g.h, g.probs, 9, v, w, debug={"moves": moves} if debug else None)
            got.append((status_of(sl.sl_mesh_status, g.h), w, t0_of(g.h, m.n_nodes)))
        assert got[0][0] == got[1][0], f"cap {cap}"
        outcomes.add(got[0][0])
        if got[0][0] == sl.SL_OK:
            assert bool((got[0][1] == got[1][1]).all()) and bool((got[0][2] == got[1][2]).all()), f"cap {cap}"
    assert outcomes == {sl.SL_OK, sl.SL_E_WALK_LIMIT}


@PRECISIONS
@pytest.mark.parametrize("kinds", [("rotation",), ("rotation", "zero"), ("rotation", "swirl")], ids="+".join)
@pytest.mark.parametrize("cap,records", [(2, 0), (3, 0), (2, 1)])
def test_a_steady_run_goes_on_walking_where_a_walk_gave_up(cap, records, kinds, precision):
    """A node whose walk ends at the caller's cap has no triangle yet: the next
    steps of a steady run walk on from where it stopped, as the steps of shorter
    runs do, which locate at every step."""
    b = Batch((40, 25)[:len(kinds)], precision)
    sl.sl_mesh_set_option(b.h, sl.SL_OPT_WALK_CAP, cap)
    sl.sl_mesh_set_option(b.h, sl.SL_OPT_RECORDS, records)
    probs = fields_of(kinds)
    a, ta, sa = run_from_start(b.h, probs, b.v0, (3, 3, 2), False)
    assert sa == sl.SL_E_WALK_LIMIT
    for _ in range(3):          # launched, recorded, replayed
        c, tc, sc = run_from_start(b.h, probs, b.v0, (8,), True)
        assert sc == sa and bool((ta == tc).all())
        if precision == sl.SL_FP32:
            assert bool((a == c).all())
        else:
            # 2^-43 of |V| and step as in whole runs; where a walk gave up the
            # value is extrapolated from up to 10 triangle widths away, in two
            # of the eight steps: errors grow by up to 20^2 < 2^9
            assert float((a - c).abs().max()) <= 8 * 2.0 ** -34 * float(a.abs().max())


def test_t0_calls_want_the_device_of_the_mesh():
    """As the step calls do.  (One GPU: the handle is told that it belongs to
    another one; the field's place is checked by what a step answers.)"""
    import torch
    b = Batch((12,))
    probs = fields_of(("rotation",))
    w = torch.empty_like(b.v0)
    j = t0_of(b.h, w.numel())
    # n_problems, N, Nt, precision, device
    place = ctypes.c_int.from_address(b.h + 28)
    assert place.value == torch.cuda.current_device()
    place.value += 1
    try:
        got = [status_of(sl.sl_step, b.h, probs, 0, b.v0, w), status_of(sl.sl_mesh_get_t0, b.h, j),
               status_of(sl.sl_mesh_set_t0, b.h, j), status_of(sl.sl_mesh_reset_t0, b.h)]
    finally:
        place.value -= 1
    assert got == [sl.SL_E_STATE] * 4


def kernels_of(call):
    """Names of the kernels a call launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for body in (torch.cuda.synchronize, call):       # a process's first session may record nothing
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            body()
            torch.cuda.synchronize()
    return [e.name for e in p.events()]


def test_fp32_configurations_of_a_mesh_of_several_waves():
    """Unset, a mesh of more than one wave takes 128 x 16; every configuration
    can be had by setting it, 128 x 12 among them."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes = {0: "256, 4", 1: "128, 16", 2: "128, 8", 3: "128, 9", 4: "256, 5", 5: "128, 12"}
    for M, unset in ((40, 5), (int((sms * 12 * 128) ** 0.5) + 5, 1)):
        m = si.courant_grid(M)
        g = DeviceRun(m, si.rotation_field(), 0.01, precision=sl.SL_FP32)
        v = g.to_dev(si.gaussian(m.xy))
        w = g.torch.empty_like(v)
        for c in (None, 5, 1, 0, 4):
            if c is None:
                assert sl.sl_mesh_get_option(g.h, sl.SL_OPT_CONFIG) == unset
            else:
                sl.sl_mesh_set_option(g.h, sl.SL_OPT_CONFIG, c)
                assert sl.sl_mesh_get_option(g.h, sl.SL_OPT_CONFIG) == c
            want = f"k_lean_f32<{shapes[unset if c is None else c]},"
            names = kernels_of(lambda: sl.sl_step(g.h, g.probs, 0, v, w))
            assert any(want in n for n in names), (M, c, names)


@pytest.mark.parametrize("strategy,cap", [(0, 0), (1, 0), (0, 50)])
def test_reading_and_setting_the_configurations_changes_no_launch(strategy, cap):
    """A program that saves its options and sets them again keeps its launches,
    also while they are unset."""
    m = si.grid_mesh(40, 0.25, 3)
    g = DeviceRun(m, si.rotation_field(), 0.01)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_STRATEGY, strategy)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_WALK_CAP, cap)
    v = g.to_dev(si.gaussian(m.xy))
    w = g.torch.empty_like(v)

    def steps():
        sl.sl_mesh_reset_t0(g.h)
        sl.sl_step(g.h, g.probs, 0, v, w)
        sl.sl_step(g.h, g.probs, 1, v, w)

    before = [n for n in kernels_of(steps) if "k_lean" in n]
    for option in (sl.SL_OPT_CONFIG, sl.SL_OPT_CONFIG_FIRST):
        sl.sl_mesh_set_option(g.h, option, sl.sl_mesh_get_option(g.h, option))
    assert len(before) == 2 and [n for n in kernels_of(steps) if "k_lean" in n] == before


@PRECISIONS
def test_the_tuner_times_steps_that_locate(precision):
    """With a steady field and any number of probe steps: what it chooses is for
    steps that locate; the others run in one form whatever it chooses."""
    m = si.grid_mesh(120, 0.25, 3)
    g = DeviceRun(m, si.rotation_field(), 0.01, precision=precision)
    v = g.to_dev(si.gaussian(m.xy))
    w = g.torch.empty_like(v)
    names = kernels_of(lambda: sl.sl_autotune(g.h, g.probs, 8, v, w))
    assert any("k_lean" in n for n in names) and not any("k_apply" in n for n in names)


@PRECISIONS
@pytest.mark.parametrize("steps", [4, 30])
def test_the_first_steady_run_of_a_handle_allocates_nothing(steps, precision):
    """Its weights have their room from the start: an allocation costs such a run
    more than the weights save."""
    m = si.grid_mesh(700, 0.25, 3)         # weights of 15 or 9 MiB: seen in what is free
    g = DeviceRun(m, si.rotation_field(), 0.001, precision=precision)
    v = g.to_dev(si.gaussian(m.xy))
    w = g.torch.empty_like(v)
    sl.sl_run(g.h, g.probs, 0, 1, v, w)
    before = g.torch.cuda.mem_get_info()[0]
    names = kernels_of(lambda: sl.sl_run(g.h, g.probs, 1, steps, v, w))
    assert any("k_apply" in n for n in names)
    assert g.torch.cuda.mem_get_info()[0] >= before - (4 << 20)


# Steps and runs of every route, their values and T0, and the device memory of a
# handle per node; with a library given, that one's.
WITHOUT_TABLES = """
import sys
import numpy as np
import torch
import paper_2104_09189_gb300 as sl
import sl_inputs as si
if len(sys.argv) > 2:
    sl._LIB_PATH = sys.argv[2]
out = {}
m = si.grid_mesh(90, 0.25, 3)
c = si.courant_grid(64)
for prec, dt in ((sl.SL_FP64, torch.float64), (sl.SL_FP32, torch.float32)):
    for name, mesh, f, opts in (("b", m, si.swirl_field(), {}), ("steady", m, si.rotation_field(), {}),
                                ("split", m, si.rotation_field(), {sl.SL_OPT_SPLIT: 1}),
                                ("cap", m, si.swirl_field(), {sl.SL_OPT_WALK_CAP: 40}),
                                ("a", m, si.swirl_field(), {sl.SL_OPT_STRATEGY: 1}),
                                ("direct", c, si.swirl_field(), {sl.SL_OPT_STRATEGY: 2}),
                                ("exclude", m, si.rotation_field(), {sl.SL_OPT_OUTSIDE: 1})):
        h = sl.sl_mesh_create(*sl.pack_meshes([(mesh.xy, mesh.tri)] * 2 if name != "direct" else [(mesh.xy, mesh.tri)]),
                              precision=prec)
        np_ = sl.sl_mesh_info(h)["n_problems"]
        probs = sl.problems([(f.kind, 0.05, f.packed())] * np_)
        for o, x in opts.items():
            sl.sl_mesh_set_option(h, o, x)
        v = torch.tensor(np.tile(si.gaussian(mesh.xy), np_), dtype=dt, device="cuda")
        w = torch.empty_like(v)
        for r in range(2):
            sl.sl_run(h, probs, 0, 3, v, w)
            sl.sl_run(h, probs, 3, 7, v, w)
            sl.sl_step(h, probs, 9, v, w)
            t0 = torch.empty(v.numel(), dtype=torch.int32, device="cuda")
            sl.sl_mesh_get_t0(h, t0)
            out[f"{name} {prec} {r} v"] = w.cpu().numpy()
            out[f"{name} {prec} {r} t0"] = t0.cpu().numpy()
            sl.sl_mesh_reset_t0(h)
        sl.sl_mesh_destroy(h)
m = si.courant_grid(1000)
before = torch.cuda.mem_get_info()[0]
h = sl.sl_mesh_create(*sl.pack_meshes([(m.xy, m.tri)]))
out["bytes"] = np.array((before - torch.cuda.mem_get_info()[0]) / m.n_nodes)
np.savez(sys.argv[1], **out)
"""


def test_a_device_without_room_for_the_tables(tmp_path):
    """A handle takes the tables and weights of the lean steps where memory is left
    over; without them it is as small as its mesh and every step is the full one,
    with the same results."""
    import glob
    import os
    import subprocess
    import sys

    from paper_2104_09189_gb300 import _build
    obj, lib = str(tmp_path / "api_device.o"), str(tmp_path / "libslwalk_small.so")
    nvcc = [_build._nvcc(), *_build.ARCH]
    subprocess.run([*nvcc, "-DSL_SPARE_BYTES=(1ull<<40)", "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I", _build.INCLUDE,
                    "-c", os.path.join(_build.CSRC, "api_device.cu"), "-o", obj], check=True)
    others = [o for o in glob.glob(os.path.join(_build.BUILD, "*.o")) if "api_device" not in o]
    subprocess.run([*nvcc, "-shared", "-o", lib, obj, *others, "-lpthread"], check=True)
    got = []
    for args in ((), (lib,)):
        out = str(tmp_path / f"out{len(got)}.npz")
        subprocess.run([sys.executable, "-c", WITHOUT_TABLES, out, *args], check=True, cwd=os.path.dirname(_build.INCLUDE))
        got.append(np.load(out))
    full, small = got
    # xy 16, xyq 16, xyh 8, tv and tn 48, he 96, t0 8, t0v 16; allocations come in 2 MiB
    assert float(small["bytes"]) <= 208 + 14 * 2.2 < float(full["bytes"])
    for k in full.files:
        if k == "bytes":
            continue
        if k.startswith(f"steady {sl.SL_FP64}") and k.endswith("v"):
            assert np.abs(full[k] - small[k]).max() <= 11 * 2.0 ** -43, k     # the weights' values
        elif k.startswith(f"split {sl.SL_FP64}") and k.endswith("v"):
            assert np.abs(full[k] - small[k]).max() <= 11 * 2.0 ** -43, k
        else:
            assert np.array_equal(full[k], small[k]), k
