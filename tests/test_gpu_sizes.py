"""The solve at the sizes where the substitutions, which give 32 rows to a warp, change their split: one
row more and less than a full warp's, and every number of warps, against the oracle (tolerances
rtol/atol-shaped as in test_gpu_parity.py).

The interval is one over which the solves do not amplify rounding: changes of two last bits (4.4e-16
relative) in T and Y, eight draws, move the oracle's own result by at most 2.4e-6 (Rosenbrock) and 2.3e-4
(Seulex) of the tolerance at every size here. The device's rates differ by a few of these, which leaves a
factor of several hundred. Over 1e-11 s the Rosenbrock solve at K = 33 (a run through ignition) moves by
183 tolerances under the same changes, so that no comparison could be made there."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2105_12070_gb300 import chem, synth

pytestmark = pytest.mark.gpu

RTOL, ATOL = 1e-6, 1e-10
P = 10.0 * synth.P_ATM_PA


@pytest.mark.parametrize("K", [31, 32, 33, 63, 64, 65, 95, 96, 97])
def test_rows_per_warp(K):
    m = synth.make_mechanism(20 + K, K, 3 * K, n_elements=4, n_third_body=K // 8, n_lindemann=2, n_troe=K // 10)
    path = m.write_temp()
    mech, ora = chem.Mechanism(path), O.OracleMechanism(path)
    T, Y = synth.cells_uniform(K, K, 3, (1000.0, 1300.0))
    for solver, name in ((chem.CHEM_SOLVER_ROSENBROCK, "rosenbrock"), (chem.CHEM_SOLVER_SEULEX, "seulex")):
        To, Yo, sto, _, _ = ora.integrate(P, T, Y, 1e-12, RTOL, ATOL, nthreads=3, solver=name)
        for G in (0, 1, 2, 4, 8):
            Td, Yd = torch.from_numpy(T.copy()).cuda(), torch.from_numpy(Y.copy()).cuda()
            status = torch.zeros(3, dtype=torch.int32, device="cuda")
            try:
                chem.chem_integrate(mech, P, Td, Yd, 1e-12, RTOL, ATOL, status=status,
                                    opts=chem.default_opts(solver=solver, warps_per_cell=G))
            except chem.ChemError as e:
                assert G and "shared memory" in str(e)  # an explicit shape may not fit; the automatic one has to
                continue
            torch.cuda.synchronize()
            assert np.all(sto == 0) and torch.all(status == 0)
            assert np.all(np.abs(Td.cpu().numpy() - To) <= RTOL * np.abs(To) + ATOL), (name, G)
            assert np.all(np.abs(Yd.cpu().numpy() - Yo) <= RTOL * np.abs(Yo) + ATOL), (name, G)
