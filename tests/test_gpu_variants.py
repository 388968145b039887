"""GPU tests of the step kernels' shortcuts: the variants that count or report
(statistics, debug outputs) take the plain path of Algorithm 1, the others may
decide a sign or start a walk another way.  The located triangles and the
values must be the same, bit for bit."""
import numpy as np
import pytest

import oracle
import paper_2104_09189_gb300 as sl
import sl_inputs as si
from gpu_helpers import REL_TOL_FP64, DeviceRun

pytestmark = pytest.mark.gpu


def step_both(g, n, v):
    """One step of the plain and of the debug variant from the same state;
    returns (V, T0) of each and leaves the mesh after the step."""
    t = g.torch
    N = g.mesh.n_nodes
    start = t.empty(N, dtype=t.int32, device=g.dev)
    sl.sl_mesh_get_t0(g.h, start)
    out, t0 = [], []
    for debug in (True, False):
        sl.sl_mesh_set_t0(g.h, start)
        w = t.empty_like(v)
        moves = t.zeros(N, dtype=t.int32, device=g.dev)
        sl.sl_step(g.h, g.probs, n, v, w, debug={"moves": moves} if debug else None)
        sl.sl_mesh_status(g.h)
        j = t.empty_like(start)
        sl.sl_mesh_get_t0(g.h, j)
        out.append(w)
        t0.append(j)
    return out, t0


@pytest.mark.parametrize("M,records", [(33, 0), (150, 0), (200, 1)])
def test_feet_at_their_nodes(M, records):
    """A swirl whose time factor vanishes (t = 1/2) at a whole time level: every
    foot is its own node to within rounding, decided around the node's
    triangles; then the steps that leave from there."""
    m = si.grid_mesh(M, 0.25, 3)
    f = si.swirl_field()
    dt, n0 = 0.05, 7
    g = DeviceRun(m, f, dt, curve=sl.SL_CURVE_HILBERT)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_RECORDS, records)
    om = oracle.OracleMesh(m.xy, m.tri)
    v = g.to_dev(si.cosine_bump(m.xy))
    for n in range(n0, n0 + 5):
        before = g.from_dev(v)
        (a, b), (ja, jb) = step_both(g, n, v)
        assert bool((ja == jb).all()), f"step {n}: located triangles differ"
        assert bool((a == b).all()), f"step {n}: values differ"
        want = om.step(f.kind, f.packed(), dt, n, before)[0]
        assert np.abs(g.from_dev(b) - want).max() <= REL_TOL_FP64 * np.abs(want).max()
        v = b


FIELDS = {
    "rotation": lambda: si.rotation_field(),
    "swirl": lambda: si.swirl_field(),
    "fourier8": lambda: si.fourier8_field(4),
    "affine": lambda: si.affine_field([0.5, -0.3, 0.2, 0.1, 0.3, 0.1, 0.3, -0.1]),
}


@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("field", list(FIELDS))
@pytest.mark.parametrize("M,dt,graded", [(9, 0.31, False), (64, 0.2, True), (181, 0.011, False), (181, 0.11, True)])
def test_walks_from_the_jump_table(M, dt, graded, field, precision):
    """Feet up to half the square away start at the jump table (also on a mesh
    of a few cells, in a clipped corner and along a side)."""
    m = si.grid_mesh(M, 0.2, 5, graded=graded)
    f = FIELDS[field]()
    g = DeviceRun(m, f, dt, curve=sl.SL_CURVE_MORTON, precision=precision)
    v = g.to_dev(si.gaussian(m.xy))
    for n in range(4):
        (a, b), (ja, jb) = step_both(g, n, v)
        assert bool((ja == jb).all()), f"step {n}: located triangles differ"
        assert bool((a == b).all()), f"step {n}: values differ"
        v = b


@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
def test_feet_on_edges_and_vertices(precision):
    """On a Courant grid of 2^-k cells a dyadic translation puts every foot on a
    vertex (whole cells) or on an edge (half cells): the triangle depends on
    the walk's path, which must be the walk from T^0."""
    m = si.courant_grid(32)
    for shift in ((4.0, 6.0), (5.5, 0.0), (3.5, 3.5), (-7.0, 2.5)):
        f = si.affine_field([shift[0] / 32, 0, 0, 0, shift[1] / 32, 0, 0, 0])
        g = DeviceRun(m, f, 1.0, curve=sl.SL_CURVE_HILBERT, precision=precision)
        v = g.to_dev(si.gaussian(m.xy))
        for n in range(3):
            (a, b), (ja, jb) = step_both(g, n, v)
            assert bool((ja == jb).all()) and bool((a == b).all()), f"shift {shift}, step {n}"
            v = b


@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -8, 2.0 ** -40], ids=["unit", "2^-8", "2^-40"])
def test_exact_signs_near_a_corner(scale, precision):
    """Feet on the lines of a grid whose first cells are `scale` / 16 wide: decided
    in integers where the coordinates are multiples of 2^-62, by the expansions
    where they are not."""
    c = np.concatenate([np.arange(16) / 16.0 * scale, [1.0] if scale == 1.0 else [scale, 0.5, 1.0]])
    n = len(c)
    xy = np.stack(np.meshgrid(c, c, indexing="xy"), -1).reshape(-1, 2)
    a = (np.arange(n - 1)[:, None] * n + np.arange(n - 1)[None, :]).ravel()
    tri = np.stack([a, a + n + 1, a + n, a, a + 1, a + n + 1], 1).reshape(-1, 3).astype(np.int32)
    m = si.Mesh(M=n - 1, xy=xy, tri=tri)
    f = si.affine_field([3.5 / 16 * scale, 0, 0, 0, 2.0 / 16 * scale, 0, 0, 0])
    g = DeviceRun(m, f, 1.0, precision=precision)
    v = g.to_dev(np.sin(np.arange(n * n)))
    for k in range(2):
        (p, q), (jp, jq) = step_both(g, k, v)
        assert bool((jp == jq).all()) and bool((p == q).all()), f"step {k}"
        v = q


@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
def test_a_hop_cap_holds_without_counting(precision):
    """A cap of the caller's ends a walk that needs more hops (and its fallback)
    whether or not the step counts or reports."""
    m = si.grid_mesh(40, 0.25, 2)
    f = si.affine_field([0.02 * 10, 0, 0, 0, 0, 0, 0, 0])      # 4 cells: 8 to 10 hops
    for cap, ok in ((1, False), (2, False), (64, True)):
        g = DeviceRun(m, f, 0.5, precision=precision)
        sl.sl_mesh_set_option(g.h, sl.SL_OPT_WALK_CAP, cap)
        v = g.to_dev(si.gaussian(m.xy))
        w = g.torch.empty_like(v)
        sl.sl_step(g.h, g.probs, 0, v, w)
        if ok:
            sl.sl_mesh_status(g.h)
        else:
            with pytest.raises(sl.SLError) as e:
                sl.sl_mesh_status(g.h)
            assert e.value.status == sl.SL_E_WALK_LIMIT


@pytest.mark.parametrize("precision,records", [(sl.SL_FP64, 0), (sl.SL_FP64, 1), (sl.SL_FP32, 0)],
                         ids=["fp64", "fp64-records8", "fp32"])
def test_every_hop_cap_is_the_plain_step(precision, records):
    """Caps around the lengths of the walks: the same outcome with and without
    the counting variant, and where no walk gave up the same triangles and values
    (the fallback's choices depend on the node and the hop alone)."""
    m = si.grid_mesh(60, 0.25, 7)
    f = si.swirl_field()
    g = DeviceRun(m, f, 0.05, precision=precision)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_RECORDS, records)
    t = g.torch
    v = g.to_dev(si.cosine_bump(m.xy))
    outcomes = set()
    for cap in range(1, 13):
        sl.sl_mesh_set_option(g.h, sl.SL_OPT_WALK_CAP, cap)
        got = []
        for debug in (True, False):
            sl.sl_mesh_reset_t0(g.h)
            w = t.empty_like(v)
            moves = t.zeros(m.n_nodes, dtype=t.int32, device=g.dev)
            sl.sl_step(g.h, g.probs, 1, v, w, debug={"moves": moves} if debug else None)
            try:
                sl.sl_mesh_status(g.h)
                status = sl.SL_OK
            except sl.SLError as e:
                status = e.status
            j = t.empty(m.n_nodes, dtype=t.int32, device=g.dev)
            sl.sl_mesh_get_t0(g.h, j)
            got.append((status, w, j))
        assert got[0][0] == got[1][0], f"cap {cap}"
        outcomes.add(got[0][0])
        if got[0][0] == sl.SL_OK:
            assert bool((got[0][1] == got[1][1]).all()) and bool((got[0][2] == got[1][2]).all()), f"cap {cap}"
    assert outcomes == {sl.SL_OK, sl.SL_E_WALK_LIMIT}


def test_jump_table_of_uneven_batch():
    """Meshes of 9 to 10 000 nodes in one batch, each with a table of its own."""
    import torch
    meshes = [si.grid_mesh(M, 0.25, M) for M in (2, 99, 3, 40, 17, 5)]
    fields = [si.swirl_field(), si.rotation_field(), si.fourier8_field(1), si.rotation_field(), si.swirl_field(),
              si.fourier8_field(2)]
    no, to, xy, tri = sl.pack_meshes([(m.xy, m.tri) for m in meshes])
    probs = sl.problems([(f.kind, 0.07, f.packed()) for f in fields])
    v0 = torch.tensor(np.concatenate([si.gaussian(m.xy) for m in meshes]), dtype=torch.float64, device="cuda")
    got = []
    for cap in (0, 1 << 20):       # a cap set by the caller turns the table off
        h = sl.sl_mesh_create(no, to, xy, tri)
        try:
            sl.sl_mesh_set_option(h, sl.SL_OPT_WALK_CAP, cap)
            v, w = v0.clone(), torch.empty_like(v0)
            sl.sl_run(h, probs, 0, 6, v, w)
            t0 = torch.empty(v.numel(), dtype=torch.int32, device="cuda")
            sl.sl_mesh_get_t0(h, t0)
            got.append((v, t0))
        finally:
            sl.sl_mesh_destroy(h)
    assert bool((got[0][0] == got[1][0]).all()) and bool((got[0][1] == got[1][1]).all())


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("steps", [1, 2, 3, 4])
def test_first_and_last_steps_on_doubles(steps, split):
    """sl_run's first step reads doubles and its last one writes them, on the
    buffers the number of steps leaves to each; so do single steps.  Values of
    every magnitude come out as the (hi, lo) pairs of the steps between."""
    m = si.grid_mesh(70, 0.25, 8)
    f = si.fourier8_field(3)
    g = DeviceRun(m, f, 0.02, curve=sl.SL_CURVE_HILBERT)
    t = g.torch
    rng = np.random.default_rng(steps)
    v0 = g.to_dev(rng.standard_normal(m.n_nodes) * np.exp2(rng.integers(-90, 90, m.n_nodes)))
    v0[:4] = t.tensor([0.0, -0.0, 1e-300, -1e300], dtype=t.float64)
    # every step through the value conversions: single split steps
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_SPLIT, 1)
    start = t.empty(m.n_nodes, dtype=t.int32, device=g.dev)
    sl.sl_mesh_get_t0(g.h, start)
    for initial in (True, False):
        ref, w = v0.clone(), t.empty_like(v0)
        sl.sl_mesh_set_t0(g.h, start)          # no longer "initial": split from the first step
        for n in range(steps):
            sl.sl_step(g.h, g.probs, n, ref, w)
            ref, w = w, ref
        sl.sl_mesh_set_option(g.h, sl.SL_OPT_SPLIT, split)
        (sl.sl_mesh_reset_t0(g.h) if initial else sl.sl_mesh_set_t0(g.h, start))
        v, w = v0.clone(), t.empty_like(v0)
        sl.sl_run(g.h, g.probs, 0, steps, v, w)
        assert np.array_equal(v.cpu().numpy().view(np.int64), ref.cpu().numpy().view(np.int64))
        (sl.sl_mesh_reset_t0(g.h) if initial else sl.sl_mesh_set_t0(g.h, start))
        v, w = v0.clone(), t.empty_like(v0)
        for n in range(steps):
            sl.sl_step(g.h, g.probs, n, v, w)
            v, w = w, v
        assert np.array_equal(v.cpu().numpy().view(np.int64), ref.cpu().numpy().view(np.int64))
        sl.sl_mesh_set_option(g.h, sl.SL_OPT_SPLIT, 1)


def test_single_steps_of_a_batch_follow_their_constants():
    """A batch of more problems than one launch of constants takes, stepped
    without a synchronisation in between."""
    import torch
    meshes = [si.grid_mesh(3 + k % 9, 0.25, k) for k in range(70)]
    fields = [si.rotation_field(1.0 + 0.1 * k) for k in range(70)]
    no, to, xy, tri = sl.pack_meshes([(m.xy, m.tri) for m in meshes])
    probs = sl.problems([(f.kind, 0.05, f.packed()) for f in fields])
    v0 = torch.tensor(np.concatenate([si.gaussian(m.xy) for m in meshes]), dtype=torch.float64, device="cuda")
    h = sl.sl_mesh_create(no, to, xy, tri)
    try:
        v, w = v0.clone(), torch.empty_like(v0)
        sl.sl_run(h, probs, 0, 5, v, w)
        sl.sl_mesh_reset_t0(h)
        a, b = v0.clone(), torch.empty_like(v0)
        for n in range(5):
            sl.sl_step(h, probs, n, a, b)
            a, b = b, a
        # pairs between the steps of a run, doubles between single steps: 48 bits
        assert float((a - v).abs().max()) <= 5 * 2.0 ** -46
    finally:
        sl.sl_mesh_destroy(h)


STEADY = {
    "rotation": lambda: si.rotation_field(),
    "zero": lambda: si.zero_field(),
    "affine": lambda: si.affine_field([0.5, -0.3, 0.2, 0.0, 0.3, 0.1, 0.3, 0.0]),
}


def runs_of(h, probs, v0, chunks):
    """The values and T0 after runs of the given numbers of steps."""
    import torch
    v, w = v0.clone(), torch.empty_like(v0)
    sl.sl_mesh_reset_t0(h)
    n = 0
    for c in chunks:
        sl.sl_run(h, probs, n, c, v, w)
        n += c
    t0 = torch.empty(v.numel(), dtype=torch.int32, device="cuda")
    sl.sl_mesh_get_t0(h, t0)
    return v, t0


@pytest.mark.parametrize("precise", [0, 1, 32])
@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("field", list(STEADY))
def test_steady_fields_keep_their_weights(field, precision, split, precise):
    """Runs of 4 steps and more of a steady field store the weights at the first
    step; runs of 3 and fewer locate at every step.  (Feet that are their
    nodes, clipped feet and steep data included.)"""
    m = si.grid_mesh(75, 0.25, 9)
    g = DeviceRun(m, STEADY[field](), 0.05, curve=sl.SL_CURVE_HILBERT, precision=precision)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_SPLIT, split)
    sl.sl_mesh_set_option(g.h, sl.SL_OPT_PRECISE, precise)
    rng = np.random.default_rng(1)
    v0 = g.to_dev(si.gaussian(m.xy) + 1e-3 * rng.standard_normal(m.n_nodes))
    a, ta = runs_of(g.h, g.probs, v0, (3, 3, 1))
    for chunks in ((7,), (4, 3), (2, 5)):
        b, tb = runs_of(g.h, g.probs, v0, chunks)
        assert bool((ta == tb).all())
        if precision == sl.SL_FP32:
            assert bool((a == b).all())
        else:
            # one step: theta_k within 2^-44 and the sums within 2^-46 of |V|, an
            # interpolation of the errors before it; between runs also the 48
            # bits of a pair
            assert float((a - b).abs().max()) <= 7 * 2.0 ** -43 * float(v0.abs().max())


@pytest.mark.parametrize("precision", [sl.SL_FP64, sl.SL_FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("kinds", [("rotation", "swirl", "zero", "affine"), ("rotation", "zero", "affine", "rotation")])
def test_batch_of_steady_and_other_fields(kinds, precision):
    import torch
    fields = [STEADY[k]() if k in STEADY else si.swirl_field() for k in kinds]
    meshes = [si.grid_mesh(M, 0.25, M) for M in (31, 64, 2, 45)]
    no, to, xy, tri = sl.pack_meshes([(m.xy, m.tri) for m in meshes])
    probs = sl.problems([(f.kind, 0.04, f.packed()) for f in fields])
    dt = torch.float64 if precision == sl.SL_FP64 else torch.float32
    v0 = torch.tensor(np.concatenate([si.gaussian(m.xy) for m in meshes]), dtype=dt, device="cuda")
    h = sl.sl_mesh_create(no, to, xy, tri, precision=precision)
    try:
        a, ta = runs_of(h, probs, v0, (3, 3, 2))
        for split in (0, 1):
            sl.sl_mesh_set_option(h, sl.SL_OPT_SPLIT, split)
            for _ in range(3):      # launched, recorded, replayed
                b, tb = runs_of(h, probs, v0, (8,))
                assert bool((ta == tb).all())
                assert float((a - b).abs().max()) <= (8 * 2.0 ** -43 if precision == sl.SL_FP64 else 0.0)
    finally:
        sl.sl_mesh_destroy(h)
