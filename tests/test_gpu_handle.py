"""GPU tests of what a mesh handle keeps between calls: recorded graphs and
their constants, steady weights, T^0, options, the tuner, device memory."""
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
