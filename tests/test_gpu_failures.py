"""Failure detection on the GPU without a GPU fault.

The tiled kernels wait for their tile copies with bounded waits and latch
SWE_ETIMEOUT when a wait runs out (instead of hanging). A mesh built with
swe_params.wait_rounds = -1 makes the first wait of every step give up at
once, so the timeout path runs deterministically: the copies already in
flight are still waited for (with the normal limit) before each block
exits, the step reports SWE_ETIMEOUT, later steps are skipped, and the
device stays usable: a fresh state on the same device then steps and
matches the oracle.
"""
import numpy as np
import pytest

from paper_1807_00672_gb300 import inputs, swe

from gpu_util import ensure_built, field_errors, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,sched", [("f64", 0), ("f32", 0), ("f32", 1)])
def test_wait_that_runs_out_reports_timeout_and_device_recovers(prec, sched):
    ensure_built()
    case = inputs.random_flow_case(nx=37, ny=23, seed=41)   # 1,702 cells, several tiles
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, kernel="tiled", tile=128,
                    halo_schedule=sched, wait_rounds=-1)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)  # init has no waits
    h0, _, _ = st.fields()
    with pytest.raises(swe.SweError) as ei:
        st.step()
    assert ei.value.status == swe.SWE_ETIMEOUT
    # later steps are skipped: the error stays latched, the clock stays at 0
    st.run(20, sync=False)
    with pytest.raises(swe.SweError) as ei:
        st.sync()
    assert ei.value.status == swe.SWE_ETIMEOUT
    info = st.info()
    assert info["err"] & 4 and info["steps"] <= 1
    st.close()
    mesh.close()

    # the device is still usable: a fresh mesh and state with the default limit
    ref, _ = oracle_run(case, 20)
    mesh2 = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, kernel="tiled", tile=128,
                     halo_schedule=sched)
    st2 = swe.State(mesh2, case.h, case.hu, case.hv, case.z, case.n)
    st2.run(20)
    if prec == "f64":
        errs, _ = field_errors(st2, ref)
        assert max(errs.values()) <= 1e-11, errs
    else:
        h, _, _ = st2.fields()
        assert np.abs(h - ref.h).max() <= 1e-4 * np.abs(ref.h).max()
    assert st2.info()["err"] == 0


def test_gradient_recording_reports_timeout():
    ensure_built()
    case = inputs.random_flow_case(nx=20, ny=12, seed=7)
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision="f64", tile=128, wait_rounds=-1)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    with pytest.raises(swe.SweError) as ei:
        swe.Tape(st, 5, 2, [0, 3])
    assert ei.value.status == swe.SWE_ETIMEOUT


@pytest.mark.parametrize("kernel", ["tiled", "edge"])
def test_negative_input_depths_are_clipped_and_counted(kernel):
    """A negative depth injected into the initial state is not a fault: the
    first step clips it at 0 and counts it (swe_state_info), as the oracle
    does; the state then matches the oracle's to 1e-11 and stays >= 0."""
    ensure_built()
    case = inputs.random_flow_case(nx=37, ny=23, seed=41)
    # a dry disc (no inflow within 10 steps) whose inner cells hold -1 cm
    c = inputs.centroids(case.mesh)
    r = np.hypot(c[:, 0] - 60.0, c[:, 1] - 40.0)
    for f in (case.h, case.hu, case.hv):
        f[r < 40.0] = 0.0
    case.h[r < 15.0] = -0.01
    ref, _ = oracle_run(case, 10)
    assert ref.neg == int((case.h < 0).sum()) > 0
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision="f64", kernel=kernel)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    st.run(10)
    info = st.info()
    assert info["neg"] == ref.neg and info["err"] == 0
    errs, (h, _, _) = field_errors(st, ref)
    assert max(errs.values()) <= 1e-11, errs
    assert np.all(h >= 0.0)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("kernel", ["tiled", "edge", "auto"])
def test_a_rate_that_overflows_is_an_error(kernel, prec):
    """Momentum whose square overflows, in a dry cell that the first step
    wets: the CFL rate is infinite and the next time step would be 0, at this
    and every later step. The step latches SWE_ENAN; advance ends with it."""
    ensure_built()
    case = inputs.random_flow_case(nx=37, ny=23, seed=41)
    assert case.h[100] == 0.0
    case.hu[100] = 1e30 if prec == "f32" else 1e200
    case.n[:] = 0.0
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, kernel=kernel)
    for call in (lambda st: st.run(30), lambda st: st.advance(1e3)):
        st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
        with pytest.raises(swe.SweError) as ei:
            call(st)
        assert ei.value.status == swe.SWE_ENAN
        assert st.info()["err"] == 1


@pytest.mark.parametrize("kernel", ["tiled", "edge", "auto"])
def test_advance_to_a_time_already_reached(kernel):
    """No step, the state as it was, and later steps as if nothing had been
    asked; with an error latched, that error."""
    ensure_built()
    case = inputs.random_flow_case(nx=37, ny=23, seed=41)
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision="f64", kernel=kernel)
    a, b = (swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n) for _ in range(2))
    for st in (a, b):
        st.run(10)
    t = a.t
    for end in (t, 0.5 * t, 0.0, -1.0, -np.inf):
        assert a.advance(end) == 0 and a.t == t and a.info()["steps"] == 10
    for st in (a, b):
        st.run(5)
        assert st.advance(3.0 * t) > 0 and st.t == 3.0 * t
    for x, y in zip(a.fields(), b.fields()):
        assert np.array_equal(x, y)
    case.hu[100] = 1e200
    case.n[:] = 0.0
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    for end in (1e3, 0.0, 1e3):
        with pytest.raises(swe.SweError) as ei:
            st.advance(end)
        assert ei.value.status == swe.SWE_ENAN
