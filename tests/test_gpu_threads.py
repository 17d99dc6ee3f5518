"""Handles of different sizes used by several host threads at once: the launches of one kernel with
different amounts of shared memory do not get into each other's way."""
import threading

import numpy as np
import pytest

from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


@pytest.mark.parametrize("dtype", ["r32", "r64"])
def test_threads_with_handles_of_different_sizes(dtype):
    """Block-form sweeps, both expectation families and the row 1-RDM, three sizes at once: every call
    returns what the handle's first, undisturbed one did."""
    tol = 1e-5 if dtype == "r32" else 1e-9   # the parity suite's gradient tolerance
    failures, jobs = [], []
    for n, ne in ((8, 2), (14, 4), (18, 8), (22, 8)):
        p = inputs.make_problem(n, ne, 20, seed=n)
        ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
        st = sv.StateVector(n, dtype, sector=(ne // 2, ne // 2))
        st.prepare_hf(p["occ"])
        E, g = st.energy_grad(ham, p["ops"], p["theta"])
        jobs.append((st, ham, p, E, g, st.rdm1()))

    def work(st, ham, p, E, g, rdm):
        try:
            for k in range(2000):
                if k % 10 == 0:
                    E2, g2 = st.energy_grad(ham, p["ops"], p["theta"])
                    assert abs(E2 - E) <= tol and np.max(np.abs(g2 - g)) <= tol
                assert np.max(np.abs(st.rdm1() - rdm)) <= tol
        except Exception as e:  # noqa: BLE001 -- handed to the main thread
            failures.append((p["n_qubits"], repr(e)))

    threads = [threading.Thread(target=work, args=job) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    for st, ham, *_ in jobs:
        st.close()
        ham.close()
