"""Scheduling options of chem_integrate (the GPU counterpart of the paper's load balancing,
Sec. 2.2): results do not depend on how cells are scheduled, and the graph and batch paths give
the same answer as the plain launch."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2105_12070_gb300 import autotune, chem, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    w = synth.workload_small()
    return w, chem.Mechanism(w["mech"].write_temp())


def _run(mech, w, opts, T=None, Y=None):
    T = torch.from_numpy((w["T"] if T is None else T).copy()).cuda()
    Y = torch.from_numpy(np.ascontiguousarray(w["Y"] if Y is None else Y)).cuda()
    st = chem.chem_integrate(mech, w["p_Pa"], T, Y, w["dt"], w["rtol"], w["atol"], opts=opts, want_stats=True)
    torch.cuda.synchronize()
    return T.cpu().numpy(), Y.cpu().numpy(), st


def test_graph_replay_and_batches_are_bitwise_equal(small):
    w, mech = small
    ref = _run(mech, w, chem.default_opts())
    for opts in (chem.default_opts(use_graph=1), chem.default_opts(use_graph=1),  # capture, then replay
                 chem.default_opts(batch_cells=37), chem.default_opts(batch_cells=64, use_queue=0),
                 chem.default_opts(batch_cells=100, use_graph=1), chem.default_opts(warps_per_cell=8)):
        T, Y, st = _run(mech, w, opts)
        np.testing.assert_array_equal(T, ref[0])
        np.testing.assert_array_equal(Y, ref[1])
        assert (st.steps, st.rejects) == (ref[2].steps, ref[2].rejects)


def test_graph_recaptures_on_new_arguments(small):
    w, mech = small
    a = _run(mech, w, chem.default_opts(use_graph=1), T=w["T"][:100], Y=w["Y"][:, :100])
    b = _run(mech, w, chem.default_opts(use_graph=1), T=w["T"][:50], Y=w["Y"][:, :50])
    c = _run(mech, w, chem.default_opts(), T=w["T"][:50], Y=w["Y"][:, :50])
    np.testing.assert_array_equal(b[0], c[0])
    np.testing.assert_array_equal(a[0][:50], c[0])


def test_autotune_returns_a_valid_shape(small, tmp_path):
    w, mech = small
    opts = autotune.autotune(mech, w["p_Pa"], w["T"], w["Y"], w["dt"], cache_path=str(tmp_path / "c.json"))
    assert opts.warps_per_cell in (1, 2, 4, 8) and opts.cells_per_cta >= 1
    again = autotune.autotune(mech, w["p_Pa"], w["T"], w["Y"], w["dt"], cache_path=str(tmp_path / "c.json"))
    assert (again.warps_per_cell, again.cells_per_cta) == (opts.warps_per_cell, opts.cells_per_cta)
    T, Y, st = _run(mech, w, opts)
    ref = _run(mech, w, chem.default_opts())
    np.testing.assert_array_equal(T, ref[0])


def test_uneven_field_mech100_parity_and_order_independence():
    """100 species / 700 reactions: sampled igniting, cold and burnt cells match the oracle, and
    the blocked and shuffled orders give each cell the same result."""
    w = synth.workload_uneven(200, "blocked")
    path = w["mech"].write_temp()
    mech = chem.Mechanism(path)
    ora = O.OracleMechanism(path)
    cls = w["cls"]
    idx = np.concatenate([np.where(cls == c)[0][:3] for c in (0, 1, 2)])
    T, Y = w["T"][idx], w["Y"][:, idx]
    Tg, Yg, st = _run(mech, w, chem.default_opts(), T=T, Y=Y)
    To, Yo, so, _, _ = ora.integrate(w["p_Pa"], T, Y, w["dt"], w["rtol"], w["atol"], nthreads=16)
    assert st.failed_cells == 0 and np.all(so == 0)
    assert np.all(np.abs(Tg - To) <= 1e-6 * np.abs(To) + 1e-10)
    assert np.all(np.abs(Yg - Yo) <= 1e-6 * np.abs(Yo) + 1e-10)
    # the same cells in another position of a larger, reordered field give the same result
    perm = np.random.default_rng(1).permutation(200)
    Tall, Yall, st2 = _run(mech, w, chem.default_opts(), T=w["T"][perm], Y=w["Y"][:, perm])
    inv = np.argsort(perm)
    np.testing.assert_array_equal(Tall[inv][idx], Tg)


@pytest.mark.parametrize("solver,dt,max_steps", [(chem.CHEM_SOLVER_ROSENBROCK, 1e-10, 3000),
                                                 (chem.CHEM_SOLVER_SEULEX, 1e-6, 600)])
def test_cells_beside_each_other_do_not_matter(solver, dt, max_steps):
    """The warps of a cell meet only at their group's barrier: with one to five cells on an SM, whose
    timing differs, every cell has the same bits."""
    w = synth.workload_shear_layer(32)
    mech = chem.Mechanism(w["mech"].write_temp())
    idx = np.arange(0, 1024, 5)
    ref = None
    for cpc in (1, 2, 3, 4, 5):
        T = torch.from_numpy(w["T"][idx].copy()).cuda()
        Y = torch.from_numpy(np.ascontiguousarray(w["Y"][:, idx])).cuda()
        opts = chem.default_opts(solver=solver, max_steps=max_steps, cells_per_cta=cpc, warps_per_cell=2)
        st = chem.chem_integrate(mech, w["p_Pa"], T, Y, dt, w["rtol"], w["atol"], opts=opts, want_stats=True)
        got = (st.steps, st.rejects, T, Y)
        assert st.failed_cells == 0
        if ref is None:
            ref = got
        assert got[:2] == ref[:2] and torch.equal(T, ref[2]) and torch.equal(Y, ref[3]), cpc


@pytest.mark.parametrize("solver", [chem.CHEM_SOLVER_ROSENBROCK, chem.CHEM_SOLVER_SEULEX])
def test_warps_per_cell_keep_the_bits(solver):
    """From 32 to 64 species every thread holds at most one component with 2, 4 or 8 warps: the automatic
    shape may take more warps for a call of few cells without changing a cell's result."""
    w = synth.workload_shear_layer(16)
    mech = chem.Mechanism(w["mech"].write_temp())
    idx = np.arange(0, 256, 37)
    ref = None
    for shape in (dict(warps_per_cell=2), dict(warps_per_cell=4), dict(warps_per_cell=8), dict()):
        T = torch.from_numpy(w["T"][idx].copy()).cuda()
        Y = torch.from_numpy(np.ascontiguousarray(w["Y"][:, idx])).cuda()
        chem.chem_integrate(mech, w["p_Pa"], T, Y, 1e-9, w["rtol"], w["atol"],
                            opts=chem.default_opts(solver=solver, **shape))
        torch.cuda.synchronize()
        if ref is None:
            ref = (T, Y)
        assert torch.equal(T, ref[0]) and torch.equal(Y, ref[1]), shape


class _Side(ctypes.Structure):
    _fields_ = [("mech", ctypes.c_void_p), ("T", ctypes.c_void_p), ("Y", ctypes.c_void_p), ("n", ctypes.c_int64),
                ("J", ctypes.c_void_p), ("stream", ctypes.c_void_p)]


def test_two_threads_with_their_own_handles(tmp_path):
    """Two host threads, each with a handle of the same mechanism and a stream of its own, one with five
    cells on an SM and one with three: the kernel's shared-memory limit, which belongs to the process, has to
    hold for both."""
    lib = str(tmp_path / "two_threads.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", lib,
                    os.path.join(os.path.dirname(os.path.abspath(__file__)), "two_threads.cpp"), "-lpthread"], check=True)
    fn = ctypes.CDLL(lib).two_threads
    fn.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    path = synth.mechanism_53().write_temp()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    keep, sides = [], []
    for n in (5 * sms, 3 * sms):  # (the same kernel: 2 warps per cell)
        mech, stream = chem.Mechanism(path), torch.cuda.Stream()
        T, Y = synth.cells_uniform(1, mech.K, n, (1000.0, 1300.0))
        T, Y = torch.from_numpy(T).cuda(), torch.from_numpy(np.ascontiguousarray(Y)).cuda()
        J = torch.full((n, mech.N, mech.N), float("nan"), dtype=torch.float64, device="cuda")
        keep.append((mech, stream, T, Y, J))
        sides.append(_Side(mech.handle, T.data_ptr(), Y.data_ptr(), n, J.data_ptr(), stream.cuda_stream))
    torch.cuda.synchronize()
    jacobian = ctypes.cast(chem.load_library().chem_jacobian, ctypes.c_void_p)
    failed = fn(jacobian, 1e6, ctypes.addressof(sides[0]), ctypes.addressof(sides[1]), 4000)
    torch.cuda.synchronize()
    assert failed == 0
    assert all(torch.isfinite(k[4]).all() for k in keep)
