"""The positivity scaling (Zhang-Shu type factors of the nodal and the point states) of
every predictor schedule and form, on a rough state that needs it in most zones, on
meshes whose zones do not fill the last block (of 4, 8 or 16 zones) and whose blocks span
columns.

FP64: the schedules run the same arithmetic in another order, 1e-12 per variable.
FP32-bulk: the point states themselves are compared (the scaling takes pressures down to
1e-13, which FP32 cannot hold against the energy, so the solvers behind it break down on
this state in every schedule).  The schedules are roundings of the same arithmetic there:
per variable the one is no further from the FP64 states than 4 times the other, or than
2e-5 (the form's documented error); the sums run over thousands of points.  At order 4 the
FP32 Picard iteration itself overflows where a nodal density is taken to 1e-13, so the state
is rough in the pressure and has 1/10 of a decade in the density."""
import numpy as np
import pytest

from conftest import gpu_available
from test_gpu_parity import rel_l1, rough_state

pytestmark = pytest.mark.gpu
MESHES = [(5, 3, 2), (3, 7, 2), (5, 3, 3), (3, 5, 3), (3, 5, 4), (3, 7, 4), (5, 3, 4)]


@pytest.fixture(autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")


def rough_pressure(U, seed=7):
    """As rough_state, with the density over 0.1 decades and the pressure over 0.6."""
    from paper_1905_02504_gb300.inputs import uniform_pm1
    u = uniform_pm1(np.arange(4 * len(U)), seed=seed).reshape(4, len(U))
    rho, p = 10.0 ** (0.1 * u[0] - 0.1), 10.0 ** (0.6 * u[1] - 0.6)
    v, B = 0.5 * np.stack([u[2], u[3], u[2] * u[3]], 1), U[:, 5:8]
    E = p / (2.0 / 3.0) + 0.5 * rho * (v * v).sum(1) + 0.5 * (B * B).sum(1)
    return np.concatenate([rho[:, None], rho[:, None] * v, E[:, None], B], 1)


def rough(n, nr, p, state=rough_state):
    from paper_1905_02504_gb300 import geomhd
    from paper_1905_02504_gb300.inputs import make_problem
    m = geomhd.Mesh(n, nr, 1.0, 2.0, p)
    U, phi = m.initial_state(make_problem("smooth"), nq_zone=3, nq_edge=4)
    U = np.ascontiguousarray(state(U.T).T)
    m.upload(U, phi)
    dt = m.cfl_dt(0.3)
    m.close()
    return U, phi, dt


def with_mesh(n, nr, p, prec, positivity, schedule, U, phi, fn):
    from paper_1905_02504_gb300 import geomhd
    m = geomhd.Mesh(n, nr, 1.0, 2.0, p, prec=prec)
    geomhd.geo_set_predictor(m.h, schedule)
    geomhd.geo_set_positivity(m.h, positivity)
    m.upload(U, phi)
    out = fn(m)
    m.close()
    return out


@pytest.mark.parametrize("schedule", [2, 1])
@pytest.mark.parametrize("n,nr,p", MESHES)
def test_step_is_the_same_in_every_schedule(n, nr, p, schedule):
    U, phi, dt = rough(n, nr, p)

    def step(m):
        m.step(dt)
        return m.download()

    ref, pref = with_mesh(n, nr, p, 0, 1, 0, U, phi, step)
    a, pa = with_mesh(n, nr, p, 0, 1, schedule, U, phi, step)
    assert np.all(rel_l1(a, ref, axis=-1) <= 1e-12) and rel_l1(pa, pref) <= 1e-12
    off, _ = with_mesh(n, nr, p, 0, 0, schedule, U, phi, step)
    moved = ~np.all(np.abs(off - ref) <= 1e-3 * np.abs(ref).max(axis=-1, keepdims=True), axis=0)
    assert moved.mean() > 0.2  # without the scaling, many zones end elsewhere


@pytest.mark.parametrize("schedule", [2, 1])
@pytest.mark.parametrize("n,nr,p", MESHES)
def test_point_states_are_scaled_alike_in_fp32(n, nr, p, schedule):
    from paper_1905_02504_gb300 import geomhd
    U, phi, dt = rough(n, nr, p, rough_state if p < 4 else rough_pressure)
    nqt, ns = {2: (24, 1), 3: (24, 2), 4: (42, 3)}[p]

    def states(m):
        for s in range(3):
            geomhd.geo_debug_run_stage(m.h, s, dt)
        out = [geomhd.geo_debug_buffer(m.h, w, (p - 1) * k * 8 * m.Z).reshape((p - 1) * k, 8, m.Z)
               for w, k in ((2, nqt), (3, 12 * ns))]
        return np.concatenate(out).transpose(1, 0, 2).reshape(8, -1)

    ref = with_mesh(n, nr, p, 0, 1, 0, U, phi, states)
    one = with_mesh(n, nr, p, 1, 1, 0, U, phi, states)
    got = with_mesh(n, nr, p, 1, 1, schedule, U, phi, states)
    off = with_mesh(n, nr, p, 1, 0, schedule, U, phi, states)
    err, bound = rel_l1(got, ref, axis=-1), np.maximum(4.0 * rel_l1(one, ref, axis=-1), 2e-5)
    assert np.all(err <= bound), (err, bound)
    # and the scaling acted, in many zones
    moved = np.abs(off - got) > 1e-3 * np.abs(ref).mean(axis=-1, keepdims=True)
    assert moved.reshape(8, -1, len(U[0])).any(axis=(0, 1)).mean() > 0.1
