"""Meshes whose tile shape is left to the library and that fit in the chip's
shared memory take the resident kernel (many steps per launch). Its results
are those of the one-step tiled kernel (the same arithmetic per face and
cell, and the same dt sequence): equal bit for bit, over sizes from one cell
to the largest that fits, both precisions, every cell order, ensembles, the
depth residual, any split of a run into calls, and end times."""
import os
import shutil
import subprocess
import threading

import numpy as np
import pytest

import oracle
from paper_1807_00672_gb300 import inputs, swe

from gpu_util import ensure_built, field_errors, oracle_run

pytestmark = pytest.mark.gpu


def pair(case, prec, order="morton", residual=False, tile=256):
    ensure_built()
    out = []
    for kw in (dict(), dict(kernel="tiled", tile=tile)):
        mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, order=order,
                        compensated_depth=residual, **kw)
        out.append(swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n))
    return out


def assert_same(a, b, what=""):
    for name, x, y in zip(("h", "hu", "hv"), a.fields(), b.fields()):
        assert np.array_equal(x, y), (what, name, np.abs(x - y).max())
    assert a.info() == b.info(), what
    assert a.next_dt() == b.next_dt() and a.t == b.t, what


def small_case(nx, ny, seed):
    return inputs.random_flow_case(nx=nx, ny=ny, lx=10.0 * nx, ly=10.0 * ny, seed=seed,
                                   jitter=0.3 if min(nx, ny) > 1 else 0.0)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 7), (9, 5), (33, 23), (151, 8), (97, 101)])
def test_same_bits_as_the_tiled_step(prec, nx, ny):
    a, b = pair(small_case(nx, ny, 3 + nx), prec)
    for n in (1, 2, 17, 40):
        a.run(n)
        b.run(n)
        assert_same(a, b, (nx, ny, n))
    assert a.step() == b.step()
    assert_same(a, b)


@pytest.mark.parametrize("prec,nx,ny", [("f64", 410, 205), ("f32", 560, 280), ("f64", 420, 211),
                                        ("f32", 570, 291), ("f64", 300, 131)])
def test_same_bits_at_the_largest_sizes(prec, nx, ny):
    a, b = pair(small_case(nx, ny, 5), prec)
    a.run(12)
    b.run(12)
    assert_same(a, b)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("order", ["none", "rcm"])
def test_other_cell_orders(prec, order):
    case = inputs.humps_case(nx=61, ny=33, lx=2_000.0, ly=1_000.0, seed=45)
    a, b = pair(case, prec, order)
    a.run(60)
    b.run(60)
    assert_same(a, b, order)
    assert a.mass == pytest.approx(b.mass, rel=1e-13 if prec == "f64" else 1e-7)


def test_depth_residual():
    a, b = pair(inputs.water_drop_case(n=71), "f32", residual=True, tile=512)
    for n in (1, 50):
        a.run(n)
        b.run(n)
        assert_same(a, b)
    assert a.mass == pytest.approx(b.mass, rel=1e-12)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_end_times(prec):
    """advance to an end time, in pieces and past it, and a run after it."""
    a, b = pair(inputs.three_mounds_case(nx=60, ny=24), prec)
    assert a.advance(0.31) == b.advance(0.31) > 1
    assert a.t == 0.31
    assert_same(a, b)
    assert a.advance(0.31) == 0
    assert a.advance(0.8) == b.advance(0.8)
    a.run(3)
    b.run(3)
    assert_same(a, b)
    case = inputs.stoker_case()
    ref = oracle.state_from_case(case)
    k = ref.advance(2.0)
    st = pair(case, "f64")[0]
    assert st.advance(2.0) == k and st.t == 2.0
    assert max(field_errors(st, ref)[0].values()) <= 1e-11


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_ensembles_and_scenarios_that_stop_apart(prec):
    ensure_built()
    cases = [inputs.stoker_case(nx=10 + 13 * i, ny=3 + 2 * i, lx=20.0 + 9 * i, seed=i) for i in range(5)]
    cat = lambda f: np.concatenate([getattr(c, f) for c in cases])
    sts = []
    for kw in (dict(), dict(kernel="tiled", tile=128)):
        mesh = swe.Mesh.ensemble([(c.mesh.xy, c.mesh.tri) for c in cases], precision=prec, **kw)
        sts.append(swe.State(mesh, cat("h"), cat("hu"), cat("hv"), cat("z"), cat("n")))
    for st in sts:
        st.run(20)
    assert_same(*sts)
    for st in sts:
        st.advance(2.0)
    assert_same(*sts)
    for i in range(5):
        x, y = sts[0].scenario(i), sts[1].scenario(i)
        assert x.pop("mass") == pytest.approx(y.pop("mass"), rel=1e-13 if prec == "f64" else 1e-7)
        assert x == y and x["t"] == 2.0


def test_reset_states_and_two_states_on_one_mesh():
    """A state set anew after runs of any length starts clean (the exchange
    words of earlier launches are never taken for new ones)."""
    case = inputs.humps_case(nx=61, ny=33, lx=2_000.0, ly=1_000.0, seed=45)
    a, b = pair(case, "f32")
    c = swe.State(a.mesh, case.h, case.hu, case.hv, case.z, case.n)
    b.run(10)
    for n in (1, 2, 3, 10):
        a.run(n)
        c.run(3)
        a.set(case.h, case.hu, case.hv)
        a.run(10)
        assert_same(a, b, n)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_errors_are_latched(prec):
    case = inputs.random_flow_case(nx=37, ny=23, seed=41)
    ensure_built()
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, wait_rounds=-1)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    for _ in range(2):
        with pytest.raises(swe.SweError) as ei:
            st.run(5)
        assert ei.value.status == swe.SWE_ETIMEOUT
    assert st.info()["steps"] == 0
    # momentum whose square overflows: SWE_ENAN from both kernels
    case.hu[100] = 1e30 if prec == "f32" else 1e200
    case.n[:] = 0.0
    for st in pair(case, prec):
        with pytest.raises(swe.SweError) as ei:
            st.run(30)
        assert ei.value.status == swe.SWE_ENAN
    # a state set anew clears it
    ref, _ = oracle_run(inputs.random_flow_case(nx=37, ny=23, seed=41), 20)
    ok = inputs.random_flow_case(nx=37, ny=23, seed=41)
    st = pair(ok, "f64")[0]
    st.run(20)
    assert max(field_errors(st, ref)[0].values()) <= 1e-11


def test_every_launch_advances_the_epoch(tmp_path):
    """pass_entry alone (tests/resident_entry_check.cu): the epoch a launch's
    blocks read, and the one it leaves, in whatever order they start."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "resident_entry_check")
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                    os.path.join(os.path.dirname(os.path.abspath(__file__)), "resident_entry_check.cu")],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


@pytest.mark.parametrize("prec,order", [("f64", "morton"), ("f32", "morton"), ("f32", "rcm")])
@pytest.mark.parametrize("nx,ny", [(3, 2), (37, 23), (150, 75)])
def test_launches_that_give_up_leave_the_state_alone(prec, order, nx, ny):
    """Waits that run out at once: every kind of call reports SWE_ETIMEOUT,
    again after the state is set anew (which clears the error), takes no step
    and leaves the fields as they were."""
    ensure_built()
    case = inputs.random_flow_case(nx=nx, ny=ny, seed=41)
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, order=order, wait_rounds=-1)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    before = st.fields()
    dt = st.next_dt()
    for call in (lambda: st.run(5), lambda: st.step(), lambda: st.advance(1.0), lambda: st.run(5000)):
        for _ in range(2):
            with pytest.raises(swe.SweError) as ei:
                call()
            assert ei.value.status == swe.SWE_ETIMEOUT
        assert st.info() == dict(steps=0, neg=0, err=4)
        after = [np.empty(mesh.T) for _ in range(3)]
        with pytest.raises(swe.SweError):  # copies out all the same
            st.copy_out(*after)
        for a, b in zip(after, before):
            assert np.array_equal(a, b)
        st.set(case.h, case.hu, case.hv)
        assert st.info()["err"] == 0 and st.next_dt() == dt


@pytest.mark.parametrize("prec,nx,ny", [("f64", 50, 25), ("f64", 400, 205), ("f32", 71, 71),
                                        ("f32", 560, 280)])
def test_the_shortest_waits_do_not_end_a_valid_run(prec, nx, ny):
    """wait_rounds = 1: blocks that start apart, or wait for the slowest of a
    step, stay far below the limit, launch after launch."""
    case = small_case(nx, ny, 7)
    ref = pair(case, prec)[1]
    ref.run(12)
    mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec, wait_rounds=1)
    st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
    for _ in range(30):
        st.set(case.h, case.hu, case.hv)
        for n in (1, 2, 9):
            st.run(n, sync=False)
        assert_same(st, ref)


def test_states_on_streams_and_threads_of_their_own():
    """Resident launches of several states at once, small ones that share the
    SMs and large ones that take the chip in turn, from a thread each: the
    results are those of the same run alone."""
    ensure_built()
    jobs = [(small_case(nx, ny, 11 + i), prec)
            for i, (prec, nx, ny) in enumerate([("f32", 35, 30), ("f64", 25, 20), ("f32", 400, 350),
                                                ("f64", 300, 200), ("f32", 90, 60), ("f64", 60, 40)])]

    def work(job, n):
        case, prec = job
        mesh = swe.Mesh(case.mesh.xy, case.mesh.tri, precision=prec)
        st = swe.State(mesh, case.h, case.hu, case.hv, case.z, case.n)
        out = []
        for _ in range(n):
            st.set(case.h, case.hu, case.hv)
            for k in (1, 5, 40):
                st.run(k, sync=False)
            st.advance(st.t + 3.0 * st.next_dt())
            out.append((*st.fields(), st.t))
        st.close()
        mesh.close()
        return out

    want = [work(job, 1)[0] for job in jobs]
    errors = []

    def worker(i):
        try:
            for got in work(jobs[i], 12):
                assert all(np.array_equal(a, b) for a, b in zip(got, want[i])), i
        except Exception as e:  # noqa: BLE001
            errors.append((i, e))

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
