"""The 1-RDM's row and column groups at the edges of their sizes: one and two words to a string,
a last group that is not full, a spin without pairs (empty, full, one electron), unequal spins."""
import numpy as np
import pytest

import oracle
from oracle import route_a as A
from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu

# the parity suite's 1-RDM tolerance of each precision
TOL = {"c128": 1e-12, "r64": 1e-12, "c64": 2e-6, "r32": 2e-6}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


# C(13, 6) = 1,716 strings take two words in float64, C(15, 5) = 3,003 in float32
@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("dtype", ["c128", "r64", "c64", "r32"])
@pytest.mark.parametrize("n,na,nb", [(4, 1, 0), (4, 2, 1), (6, 3, 1), (10, 2, 3), (14, 7, 1), (26, 6, 1), (30, 1, 5)])
def test_rdm_groups(n, na, nb, dtype, variant):
    rng = np.random.default_rng(100 * n + na)
    occ = [2 * p for p in range(na)] + [2 * p + 1 for p in range(nb)]
    pool = inputs.qeb_pool(n, 2 if n < 8 else 4)
    ops = pool[rng.integers(0, len(pool), 150)]
    theta = rng.normal(0, 0.7, len(ops))
    sec = oracle.Sector(n, na, nb)
    psi = A.apply_ansatz(sec, ops, theta, A.hf_state(sec, occ))
    st = sv.StateVector(n, dtype, sector=(na, nb))
    st.set_option(sv.SV_OPT_RDM_VARIANT, variant)
    st.prepare_hf(occ)
    st.apply_ansatz(ops, theta)
    assert np.max(np.abs(st.rdm1() - A.rdm1(sec, psi))) <= TOL[dtype]


def test_blocks_without_groups():
    """More blocks than row and column groups: the idle blocks add zeros, whatever shared memory held."""
    n, na, nb = 26, 6, 1
    rng = np.random.default_rng(7)
    pool = inputs.qeb_pool(n, 4)
    ops = pool[rng.integers(0, len(pool), 60)]
    theta = rng.normal(0, 0.7, len(ops))
    occ = [2 * p for p in range(na)] + [1]
    sec = oracle.Sector(n, na, nb)
    ref = A.rdm1(sec, A.apply_ansatz(sec, ops, theta, A.hf_state(sec, occ)))
    dirty = sv.StateVector(24, "r32", sector=(4, 4))  # its 1-RDM leaves other values in shared memory
    dirty.prepare_hf(list(range(8)))
    for bps in (1, 4, 16, 64):
        st = sv.StateVector(n, "r64", sector=(na, nb))
        st.set_option(sv.SV_OPT_RDM_BLOCKS_PER_SM, bps)
        st.prepare_hf(occ)
        st.apply_ansatz(ops, theta)
        for _ in range(4):
            dirty.rdm1()
            assert np.max(np.abs(st.rdm1() - ref)) <= TOL["r64"]
        st.close()


# complex amplitudes (two words to a string in float64), both sides of 64 strings (56, 70), rows left over
@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,na,nb", [(4, 2, 1), (10, 2, 3), (14, 7, 1), (16, 3, 3), (16, 4, 3), (20, 5, 4)])
def test_rdm_groups_of_complex_states(n, na, nb, dtype, variant):
    dense = inputs.random_sector_state(n, na, nb, np.random.default_rng(n + na))
    sec = oracle.Sector(n, na, nb)
    st = sv.StateVector(n, dtype, sector=(na, nb))
    st.set_option(sv.SV_OPT_RDM_VARIANT, variant)
    st.prepare_state(dense.astype(np.complex128 if dtype == "c128" else np.complex64), na, nb)
    got = st.rdm1()
    assert np.max(np.abs(got - A.rdm1(sec, dense[sec.dets.astype(np.int64)]))) <= TOL[dtype]
    assert np.max(np.abs(got.imag)) > 0.0
