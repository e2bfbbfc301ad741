"""States at the edge of the physical ones: what the FP64 arithmetic of the CFL time
step and of the state flag decides is decided in both precision forms, whatever the
kernels evaluate in FP32 first and however the state is scaled."""
import numpy as np
import pytest

from conftest import gpu_available

pytestmark = pytest.mark.gpu
GAMMA = 5.0 / 3.0


@pytest.fixture(autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")


# gamma p + B^2 below zero by a part of the energy that FP32 does not resolve, in a zone
# whose time step is not the smallest: kinetic energy alone, or with a field (then p is
# negative and B^2 makes up for all but `part` of it)
@pytest.mark.parametrize("part", [1e-6, 1e-7, 3e-8, 1e-8])
@pytest.mark.parametrize("b", [0.0, 1.0])
def test_cfl_refuses_what_fp32_cannot_tell(part, b):
    from paper_1905_02504_gb300 import geomhd
    rng = np.random.default_rng(5)
    meshes = [geomhd.Mesh(4, 8, 1.0, 2.0, 2, prec=prec) for prec in (0, 1)]
    Z = meshes[0].Z
    phi = np.zeros(meshes[0].F)
    for trial in range(24):
        U = np.zeros((8, Z))
        U[0] = 1.0
        U[1:4] = rng.normal(size=(3, 1))
        U[1:4] /= np.sqrt((U[1:4] ** 2).sum(0))
        U[4] = 0.5 + 4.0 / (GAMMA - 1.0)
        z = 8 * int(rng.integers(Z // 8)) + 7         # the outermost shell: the largest zones
        kinetic = 0.5 * (U[1:4, z] ** 2).sum() / U[0, z]
        U[5, z] = b
        b2 = b * b
        U[4, z] = (kinetic + 0.5 * b2 - b2 / (GAMMA * (GAMMA - 1.0))) - part * (kinetic + b2)
        for m in meshes:
            m.upload(U, phi)
            with pytest.raises(geomhd.GeoError):
                m.cfl_dt(0.4)
        # and accepted just above the edge, with the same time step
        U[4, z] += 2e-5 * (kinetic + b2)
        dts = []
        for m in meshes:
            m.upload(U, phi)
            dts.append(m.cfl_dt(0.4))
        assert abs(dts[1] - dts[0]) <= 1e-14 * dts[0]
    for m in meshes:
        m.close()


# density, momentum and energy times 4^k and the field times 2^k: the same flow in other
# units.  At 4^-272 the product of density and energy is below the range of FP64 (so are
# the squares of the momentum, which is why the unphysical state stops at 4^-200), at 4^250
# it is near the upper end
@pytest.mark.parametrize("k,thermal,flagged", [(-272, 1.0, False), (-200, 1.0, False), (0, 1.0, False),
                                               (250, 1.0, False), (-200, -1e-6, True), (0, -1e-6, True),
                                               (250, -1e-6, True)])
def test_state_flag_in_other_units(k, thermal, flagged):
    from paper_1905_02504_gb300 import geomhd
    from paper_1905_02504_gb300.inputs import make_problem
    m = geomhd.Mesh(3, 3, 1.0, 2.0, 2)
    U, phi = m.initial_state(make_problem("uniform", B0=(0.3, -0.2, 0.5)), nq_zone=3, nq_edge=4)
    rest = 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0] + 0.5 * (U[5] ** 2 + U[6] ** 2 + U[7] ** 2)
    U[4] = 2.0 * rest
    U[4, m.Z // 2] = rest[m.Z // 2] * (1.0 + thermal)
    s = 2.0 ** k
    U[:5] *= s * s
    U[5:] *= s
    m.upload(U, phi * s)
    m.step(1e-30)  # too short to change the state
    if flagged:
        with pytest.raises(geomhd.GeoError):
            geomhd.geo_check_state(m.h)
    else:
        geomhd.geo_check_state(m.h)
    m.close()
