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
