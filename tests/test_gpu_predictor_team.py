"""The variable-team predictor against the one-thread-per-zone schedule where its
tiles are ragged: fewer shells than zones of a block (blocks that span several
columns), last blocks that are partly empty, and both sides of every block size.

Both run the same arithmetic in another order, so one step from the same state
agrees to rounding: 1e-12 per variable in FP64 (the bound of the parity tests), 2e-5
of the whole state in the FP32-bulk form (its documented error, which both sides
carry; the momentum of a fluid starting at rest is a difference of pressures, so its
own size is no scale for FP32 rounding)."""
import numpy as np
import pytest

from conftest import gpu_available
from test_gpu_parity import rel_l1

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")


def one_step(n, nr, p, prec, positivity, schedule, problem):
    from paper_1905_02504_gb300 import geomhd
    from paper_1905_02504_gb300.inputs import make_problem
    m = geomhd.Mesh(n, nr, 1.0, 2.0, p, prec=prec)
    geomhd.geo_set_predictor(m.h, schedule)
    geomhd.geo_set_positivity(m.h, positivity)
    U, phi = m.initial_state(make_problem(problem, noise=0.01), nq_zone=3, nq_edge=4)
    m.upload(U, phi)
    dt = m.cfl_dt(0.4)
    m.step(dt)
    U1, phi1 = m.download()
    m.close()
    return U1, phi1


# 6 n^2 nr zones in blocks of 4 (order 4), 8 (order 3), 16 (order 2) zones
@pytest.mark.parametrize("positivity,problem", [(0, "smooth"), (1, "blast")])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,nr,p", [(2, 2, 2), (3, 5, 2), (2, 17, 2), (2, 2, 3), (3, 3, 3), (3, 9, 3), (2, 3, 4),
                                    (3, 3, 4), (3, 5, 4)])
def test_variable_team_matches_zone_thread(n, nr, p, prec, positivity, problem):
    a = one_step(n, nr, p, prec, positivity, 2, problem)
    b = one_step(n, nr, p, prec, positivity, 0, problem)
    if prec == 0:
        for x, y in zip(a, b):
            scale = np.abs(y).sum(axis=-1) + 1e-3 * np.abs(y).sum() / max(1, y.ndim)
            assert np.all(np.abs(x - y).sum(axis=-1) <= 1e-12 * scale)
        assert np.all(rel_l1(a[0][[0, 4]], b[0][[0, 4]], axis=-1) <= 1e-12)
    else:
        for x, y in zip(a, b):
            assert np.linalg.norm(x - y) <= 2e-5 * np.linalg.norm(y)
        assert np.all(rel_l1(a[0][[0, 4]], b[0][[0, 4]], axis=-1) <= 2e-5)
