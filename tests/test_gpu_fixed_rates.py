"""The fixed-point rate evaluation at the edges of its range, against the oracle: temperatures on both
sides of the interval it takes and of Tmid, states with zero, tiny and slightly negative mass
fractions, a species on both sides of a reaction, mechanisms it must leave to the general form, and a change of ln A that moves the
interval under a captured launch; and solves on the general form, against the oracle.  Tolerances as in
test_gpu_parity.py (1e-11 of the gross flux, 1e-12 of the row; solves rtol/atol-shaped)."""
import copy
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2105_12070_gb300 import chem, synth

pytestmark = pytest.mark.gpu

P = 5.0 * synth.P_ATM_PA
EDGES = [100.0, 159.0, 160.0, 161.0, 256.0, 256.5, 512.0, 999.9, 1000.0, 1000.1, 2999.0, 4095.0, 4097.0, 6000.0,
         8191.0, 8193.0]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _states(K, n_per_T=3, seed=5):
    rng = np.random.default_rng(seed)
    T = np.repeat(EDGES, n_per_T)
    Y = rng.dirichlet(np.ones(K), size=T.size)
    Y[::3, : K // 2] = 0.0          # absent species
    Y[1::3, 0] = 1e-30              # a trace
    Y[2::3, 1] = -1e-12             # what a transport scheme may hand over
    return T, np.ascontiguousarray(Y.T)


def _check(mech, ora, T, Y, p=P):
    f = torch.empty((mech.N, T.size), dtype=torch.float64, device="cuda")
    J = torch.empty((T.size, mech.N, mech.N), dtype=torch.float64, device="cuda")
    chem.chem_rates(mech, p, _dev(T), _dev(Y), f)
    chem.chem_jacobian(mech, p, _dev(T), _dev(Y), J)
    torch.cuda.synchronize()
    f, J = f.cpu().numpy(), J.cpu().numpy()
    fo, gross = ora.rates(p, T, Y, gross=True)
    Jo = ora.jacobian(p, T, Y)
    ok = np.isfinite(fo).all(axis=0) & np.isfinite(gross).all(axis=0) & np.isfinite(Jo).all(axis=(1, 2))
    assert ok.sum() >= T.size // 2
    assert np.all(np.abs(f - fo)[:, ok] <= 1e-11 * gross[:, ok] + 1e-300)
    rel = np.abs(J - Jo)[ok] / np.maximum(np.abs(Jo[ok]).max(axis=2, keepdims=True), 1e-300)
    assert rel.max() <= 1e-12, (rel.max(), T[ok][np.unravel_index(np.argmax(rel), rel.shape)[0]])


@pytest.mark.parametrize("make", [synth.mechanism_small, synth.mechanism_53, synth.mechanism_100])
def test_edges_of_the_range(make):
    path = make().write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = _states(mech.K)
    _check(mech, ora, T, Y)


RTOL, ATOL = 1e-6, 1e-10
SOLVERS = ((chem.CHEM_SOLVER_ROSENBROCK, "rosenbrock"), (chem.CHEM_SOLVER_SEULEX, "seulex"))


def _check_solves(mech, ora, T, Y, dt, p=P, solvers=SOLVERS, **options):
    for solver, name in solvers:
        To, Yo, sto, _, _ = ora.integrate(p, T, Y, dt, RTOL, ATOL, nthreads=4, solver=name)
        assert np.all(sto == 0)
        Td, Yd = _dev(T), _dev(Y)
        status = torch.full((T.size,), -1, dtype=torch.int32, device="cuda")
        chem.chem_integrate(mech, p, Td, Yd, dt, RTOL, ATOL, status=status,
                            opts=chem.default_opts(solver=solver, **options))
        torch.cuda.synchronize()
        assert torch.all(status == 0), (name, status)
        assert np.all(np.abs(Td.cpu().numpy() - To) <= RTOL * np.abs(To) + ATOL), name
        assert np.all(np.abs(Yd.cpu().numpy() - Yo) <= RTOL * np.abs(Yo) + ATOL), name


COLD, HOT = [100.0, 150.0, 159.0, 200.0, 250.0], [8200.0, 8500.0, 9000.0]


@pytest.mark.parametrize("make,T,dt", [(synth.mechanism_small, COLD, 1e-8), (synth.mechanism_small, HOT, 1e-10),
                                       (synth.mechanism_53, COLD, 1e-8), (synth.mechanism_100, COLD, 1e-10)])
def test_solves_outside_the_range(make, T, dt):
    """The solve keeps its state beside the evaluation's scratch: outside the interval the general form must
    stay inside it.  Changes of two last bits in T and Y (six draws) move the oracle's results by at
    most 1e-5 of the tolerance here.  (The hot cells cool to 2300-2900 K: they enter the interval on the way.)"""
    path = make().write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    rng = np.random.default_rng(5)
    Y = np.ascontiguousarray(rng.dirichlet(np.ones(mech.K), size=len(COLD) + len(HOT)).T)
    Y = np.ascontiguousarray(Y[:, :len(T)] if T is COLD else Y[:, len(COLD):])
    _check_solves(mech, ora, np.array(T), Y, dt)
    _check_solves(mech, ora, np.array(T), Y, dt, solvers=SOLVERS[:1], precision=chem.CHEM_PREC_MIXED_FF)


def test_many_reactions_outside_the_range():
    """More elementary reactions than the cell's vectors hold (R - n_pd > 12 K)."""
    m = copy.deepcopy(synth.mechanism_small())
    n_pd, copies = int((m.rtype != 0).sum()), 6
    assert np.all(m.rtype[n_pd:] == 0)
    at = np.concatenate([np.arange(n_pd)] + [np.arange(n_pd, m.R)] * copies)
    rng = np.random.default_rng(2)
    for name in ("rtype", "reac", "prod", "b", "Ea"):
        setattr(m, name, getattr(m, name)[at].copy())
    m.A = m.A[at] * rng.uniform(0.5, 2.0, at.size)
    assert m.R - n_pd > 12 * m.K
    path = m.write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = _states(mech.K)
    _check(mech, ora, T, Y)
    cold = T < 200.0
    _check_solves(mech, ora, T[cold], np.abs(Y[:, cold]), 1e-10)


def test_species_on_both_sides(tmp_path):
    """A + B = 2 B (isomers): one species in three slots of a reaction."""
    text = open(os.path.join(os.path.dirname(__file__), "golden", "isomer_AB.txt")).read()
    text = text.replace("0 1 0 -1 1 1 -1 3000.0 0.5 10000.0", "0 2 0 1 2 1 1 3e12 0.5 10000.0")
    text = text.replace("-1000.0 11.386294361119891", "-1500.0 11.386294361119891")  # a heat of reaction
    assert "0 2 0 1 2 1 1" in text and text.count("-1500.0 11.38") == 2
    path = tmp_path / "autocatalytic.txt"
    path.write_text(text)
    mech, ora = chem.Mechanism(str(path)), O.OracleMechanism(str(path))
    _check(mech, ora, *_states(mech.K))


def _outside_the_limits(m, change):
    m = copy.deepcopy(m)
    if change == "barrier":
        m.Ea[3] = 400e3     # beyond the table's 2^17 K ln 2
    elif change == "exponent":
        m.b[5] = 70.0
        m.A[5] = 1e-180
    else:
        m.A[7] = 1e290
    return m


@pytest.mark.parametrize("make,change,dt", [(synth.mechanism_small, "barrier", 1e-10), (synth.mechanism_53, "barrier", 1e-10),
                                            (synth.mechanism_53, "exponent", 1e-12)])
def test_solves_without_an_interval(make, change, dt):
    """Mechanisms that no temperature lets into fixed point, at flame temperatures.  (Two last bits in T and Y
    move the oracle's results by at most 7e-4 of the tolerance; the pre-factor's case is no solvable
    problem, nor is the exponent's with 10 species: the oracle itself fails there.)"""
    path = _outside_the_limits(make(), change).write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = synth.cells_uniform(3, mech.K, 4, (1000.0, 1300.0))
    _check_solves(mech, ora, T, Y, dt)


@pytest.mark.parametrize("change", ["barrier", "exponent", "prefactor"])
def test_mechanisms_outside_the_limits(change):
    m = _outside_the_limits(synth.mechanism_small(), change)
    path = m.write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = _states(mech.K)
    keep = (T > 200.0) & (T < 5000.0)
    T, Y = T[keep], np.ascontiguousarray(Y[:, keep])
    # one reaction may dwarf the others here: the source term against its gross flux stays meaningful
    f = torch.empty((mech.N, T.size), dtype=torch.float64, device="cuda")
    chem.chem_rates(mech, P, _dev(T), _dev(Y), f)
    torch.cuda.synchronize()
    fo, gross = ora.rates(P, T, Y, gross=True)
    ok = np.isfinite(fo).all(axis=0) & np.isfinite(gross).all(axis=0)
    assert np.all(np.abs(f.cpu().numpy() - fo)[:, ok] <= 1e-11 * gross[:, ok] + 1e-300)


def test_ln_a_change_moves_the_interval_of_a_captured_launch():
    w = synth.workload_small()
    path = w["mech"].write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    lnA = chem.chem_get_lnA(mech)
    opts = chem.default_opts(use_graph=1)
    Th, Yh = w["T"][:40], np.ascontiguousarray(w["Y"][:, :40])
    T0, Y0 = _dev(Th), _dev(Yh)
    T, Y = torch.empty_like(T0), torch.empty_like(Y0)
    status = torch.empty(40, dtype=torch.int32, device="cuda")

    def step(o, oracle):
        T.copy_(T0)
        Y.copy_(Y0)
        status.fill_(-1)
        chem.chem_integrate(mech, w["p_Pa"], T, Y, 1e-7, RTOL, ATOL, status=status, opts=o)
        torch.cuda.synchronize()
        assert torch.all(status == 0)
        To, Yo, _, _, _ = oracle.integrate(w["p_Pa"], Th, Yh, 1e-7, RTOL, ATOL, nthreads=4)
        assert np.all(np.abs(T.cpu().numpy() - To) <= RTOL * np.abs(To) + ATOL)
        assert np.all(np.abs(Y.cpu().numpy() - Yo) <= RTOL * np.abs(Yo) + ATOL)
        return T.clone(), Y.clone()

    first = step(opts, ora)
    far = lnA.copy()
    far[4] = -700.0         # a reaction switched off by its pre-factor: outside the fixed-point range
    chem.chem_set_lnA(mech, far)
    off = copy.deepcopy(w["mech"])
    off.A[4] = np.exp(-700.0)
    without = O.OracleMechanism(off.write_temp())
    replayed, direct = step(opts, without), step(chem.default_opts(), without)
    assert torch.equal(replayed[0], direct[0]) and torch.equal(replayed[1], direct[1])
    chem.chem_set_lnA(mech, lnA)
    again = step(opts, ora)
    assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])


@pytest.mark.parametrize("efficiencies", ["even", "one_hot"])
def test_third_body_sums_of_unphysical_states(efficiencies):
    """The source-term kernel's fixed-point third-body sums hand over what they cannot hold: mass
    fractions far outside [0, 1] (a diverged trial state), and mechanisms with zero efficiencies."""
    m = copy.deepcopy(synth.mechanism_53())
    if efficiencies == "one_hot":
        r = min(m.eff)
        m.eff[r] = np.eye(m.K)[3]
    path = m.write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    rng = np.random.default_rng(9)
    n = 64
    Y = rng.dirichlet(np.ones(m.K), size=n)
    for c in range(n):
        if c % 4 == 1:
            Y[c, c % m.K] -= 0.9           # one large negative, made up for elsewhere
            Y[c, (c + 7) % m.K] += 0.9
        elif c % 4 == 2:
            Y[c, ::2] += 2.0               # many beyond 1, as many below -1
            Y[c, 1::2] -= 2.0 * Y[c, ::2].size / Y[c, 1::2].size
        elif c % 4 == 3:
            Y[c, c % m.K] -= 0.03          # near the bound of 1/64 of the total
    T = rng.uniform(800.0, 2000.0, n)
    Y = np.ascontiguousarray(Y.T)
    f = torch.empty((mech.N, n), dtype=torch.float64, device="cuda")
    chem.chem_rates(mech, P, _dev(T), _dev(Y), f)
    torch.cuda.synchronize()
    fo, gross = ora.rates(P, T, Y, gross=True)
    ok = np.isfinite(fo).all(axis=0) & np.isfinite(gross).all(axis=0)
    assert ok.sum() >= n // 2
    # (a negative mean molar mass makes the density, and with it the scale, negative)
    assert np.all(np.abs(f.cpu().numpy() - fo)[:, ok] <= 1e-11 * np.abs(gross[:, ok]) + 1e-300)


def test_non_finite_fall_off_factors():
    """A negative or zero reduced pressure (a diverged trial state, an absent only collider) has no logarithm:
    the source terms that it enters are NaN, as in the oracle, and not a finite number."""
    m = copy.deepcopy(synth.mechanism_53())
    troe = [r for r in range(m.R) if m.rtype[r] == synth.TYPE_TROE]
    m.eff[troe[3]] = np.eye(m.K)[7]
    path = m.write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    X = np.ones((4, m.K))
    X[0] = 1e-3
    X[0, np.argmax(m.eff[troe[0]])], X[0, np.argmin(m.eff[troe[0]])] = -1.0, 2.0  # [M] < 0 of several reactions
    X[1, 7], X[2, 7] = 0.0, -1e-3                                                # [M] = 0 and < 0 of one
    Y = X * m.W
    Y = np.ascontiguousarray((Y / Y.sum(axis=1, keepdims=True)).T)
    T = np.full(4, 1100.0)
    f = torch.empty((mech.N, 4), dtype=torch.float64, device="cuda")
    chem.chem_rates(mech, P, _dev(T), _dev(Y), f)
    torch.cuda.synchronize()
    fo = ora.rates(P, T, Y)
    assert np.isnan(fo[:, :3]).any(axis=0).all() and np.isfinite(fo[:, 3]).all()
    np.testing.assert_array_equal(np.isnan(f.cpu().numpy()), np.isnan(fo))


@pytest.mark.parametrize("p", [1e-292, 1e-285, 1e-265, 1e-3])
def test_third_body_sums_at_tiny_pressures(p):
    """Concentrations next to the smallest normal number: the fixed-point sums hand over where their unit
    would be below it."""
    path = synth.mechanism_53().write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = synth.cells_uniform(8, mech.K, 16, (800.0, 2000.0))
    f = torch.empty((mech.N, 16), dtype=torch.float64, device="cuda")
    chem.chem_rates(mech, p, _dev(T), _dev(Y), f)
    torch.cuda.synchronize()
    fo, gross = ora.rates(p, T, Y, gross=True)
    assert np.isfinite(fo).all() and np.isfinite(gross).all() and (gross > 0).any(axis=0).all()
    assert np.all(np.abs(f.cpu().numpy() - fo) <= 1e-11 * gross + 1e-300)
