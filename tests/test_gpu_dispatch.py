"""Both sides of the rules that pick a kernel by the mesh's size.

Meshes on the large side of a rule are compared with meshes on its small side that hold
the same inner shells: the radial grid is geometric, so shells 0 .. K-1 of a mesh of nr
shells are those of a mesh of K shells whose outer radius is where shell K - 1 ends.  A
step reaches three shells, so what lies at least four below the cut agrees to rounding."""
import numpy as np
import pytest

from conftest import gpu_available

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")


def one_step(n, nr, r_out, p, prec, riemann, U, phi, dt, timing=False):
    from paper_1905_02504_gb300 import geomhd
    m = geomhd.Mesh(n, nr, 1.0, r_out, p, prec=prec)
    geomhd.geo_set_riemann(m.h, riemann)
    geomhd.geo_set_stage_timing(m.h, timing)
    m.upload(U, phi)
    m.step(dt)
    out = m.download()
    m.close()
    return out


def start(n, nr, r_out, p, problem="smooth"):
    from paper_1905_02504_gb300 import geomhd
    from paper_1905_02504_gb300.inputs import make_problem
    m = geomhd.Mesh(n, nr, 1.0, r_out, p)
    U, phi = m.initial_state(make_problem(problem, noise=0.01), nq_zone=3, nq_edge=4)
    m.upload(U, phi)
    dt = m.cfl_dt(0.4)
    m.close()
    return U, phi, dt


def close(a, b, prec):
    """Per variable: 1e-12 (the parity tests' bound), or 2e-5 of the whole state in FP32."""
    if prec:
        return np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b)
    a, b = np.atleast_2d(a), np.atleast_2d(b)
    return np.all(np.abs(a - b).sum(axis=1) <= 1e-12 * np.abs(b).sum(axis=1))


def shells(n, nr, U, phi, K):
    """State of the inner K shells: zones, radial faces, lateral faces."""
    ncol = 6 * n * n
    nrad = ncol * (nr + 1)
    Uk = U.reshape(8, ncol, nr)[:, :, :K].reshape(8, -1)
    rad = phi[:nrad].reshape(ncol, nr + 1)[:, :K + 1].ravel()
    lat = phi[nrad:].reshape(-1, nr)[:, :K].ravel()
    return np.ascontiguousarray(Uk), np.concatenate([rad, lat])


# 42,336 faces and 43,232 edges: threads per face and edge; 20,736 zones: variables per
# thread of WENO-AO; the inner 12 shells (10,368 zones) take the small side of each
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nr,p,riemann", [(16, 2, 0), (24, 2, 1), (24, 3, 0), (16, 4, 1), (24, 4, 0)])
def test_large_mesh_matches_its_inner_shells(nr, p, riemann, prec):
    n, K = 12, 12
    r_out = 2.0 ** (nr / 16.0)
    U, phi, dt = start(n, nr, r_out, p)
    Uk, pk = shells(n, nr, U, phi, K)
    a = one_step(n, nr, r_out, p, prec, riemann, U, phi, dt)
    b = one_step(n, K, r_out ** (K / nr), p, prec, riemann, Uk, pk, dt)
    a = shells(n, nr, *a, K - 4)
    b = shells(n, K, *b, K - 4)
    assert close(a[0], b[0], prec) and close(a[1], b[1], prec)


# a mesh of few faces runs its corrector in two launches, and in four when its stages are
# timed; 1,728 and 162 zones leave partly empty blocks in every part of the fused ones
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("riemann", [0, 1])
@pytest.mark.parametrize("n,nr,p", [(3, 3, 2), (6, 8, 2), (3, 3, 3), (2, 3, 4), (5, 3, 4)])
def test_fused_corrector_matches_its_stages(n, nr, p, riemann, prec):
    U, phi, dt = start(n, nr, 2.0, p)
    a = one_step(n, nr, 2.0, p, prec, riemann, U, phi, dt)
    b = one_step(n, nr, 2.0, p, prec, riemann, U, phi, dt, timing=True)
    assert close(a[0], b[0], prec) and close(a[1], b[1], prec)


# density, momentum and energy times 4^k and the field times 2^k leave every speed, and
# velocities times 2^k scale it, exactly in FP64; FP32 estimates over- or underflow on the way
@pytest.mark.parametrize("kscale,vscale", [(-74, 0), (-66, 0), (-62, 0), (-50, 0), (50, 0), (63, 0), (66, 0),
                                           (0, -80), (0, -70), (0, -66), (0, -50), (0, 50), (0, 66), (-33, -20),
                                           (-20, -33)])
def test_cfl_estimate_keeps_the_minimum(kscale, vscale):
    from paper_1905_02504_gb300 import geomhd
    U, phi, _ = start(6, 8, 2.0, 2)
    s, v = 4.0 ** kscale, 2.0 ** vscale
    scale = np.array([s] + 3 * [s * v] + [s * v * v] + 3 * [2.0 ** kscale * v])[:, None]
    dts = []
    for prec, sc, f in ((0, 1.0, 1.0), (1, scale, v)):
        m = geomhd.Mesh(6, 8, 1.0, 2.0, 2, prec=prec)
        m.upload(np.ascontiguousarray(U * sc), phi)
        dts.append(m.cfl_dt(0.4) * f)
        m.close()
    assert abs(dts[1] - dts[0]) <= 1e-14 * dts[0]


# pressures within 1e-5 of the total energy are out of reach of the FP32 test of the state
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("thermal,flagged", [(1.0, False), (5e-6, False), (-5e-6, True), (-1.0, True)])
def test_state_flag_near_vacuum(thermal, flagged, prec):
    from paper_1905_02504_gb300 import geomhd
    from paper_1905_02504_gb300.inputs import make_problem
    m = geomhd.Mesh(3, 3, 1.0, 2.0, 2, prec=prec)
    U, phi = m.initial_state(make_problem("uniform", B0=(0.3, -0.2, 0.5)), nq_zone=3, nq_edge=4)
    rest = 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0] + 0.5 * (U[5] ** 2 + U[6] ** 2 + U[7] ** 2)
    U[4] = rest * (1.0 + abs(thermal))
    z = m.Z // 2
    U[4, z] = rest[z] * (1.0 + thermal)
    m.upload(U, phi)
    m.step(1e-30)  # too short to change the state
    if flagged:
        with pytest.raises(geomhd.GeoError):
            geomhd.geo_check_state(m.h)
    else:
        geomhd.geo_check_state(m.h)
    m.close()


# timing the stages (a launch each) must not move a bit of the result; 37,500 faces and
# 41,256 edges lie on the two sides of the size rule, which goes by faces
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,nr,p", [(25, 3, 3), (3, 3, 3), (8, 8, 2), (5, 3, 4)])
def test_stage_timing_leaves_the_result_alone(n, nr, p, prec):
    U, phi, dt = start(n, nr, 2.0, p)
    a = one_step(n, nr, 2.0, p, prec, 0, U, phi, dt)
    b = one_step(n, nr, 2.0, p, prec, 0, U, phi, dt, timing=True)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
