"""The float64 expectation's integer products on the tensor cores (real float64 sectors of at least
2^12 determinants): against the oracle and the float64 sums (variant 3) at ragged string counts, at
extreme amplitude scales, under byte caps, and with a wait that runs out."""
import numpy as np
import pytest

import oracle
from oracle import route_a as A
from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu

TOL_E, TOL_G = 1e-10, 1e-9  # the parity suite's, float64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


def _problem(n, na, nb):
    rng = np.random.default_rng(n + 10 * na + nb)
    p = inputs.make_problem(n, 4, 4, seed=n)
    pool = inputs.qeb_pool(n, 4)
    ops = pool[rng.integers(0, len(pool), 80)]
    occ = [2 * k for k in range(na)] + [2 * k + 1 for k in range(nb)]
    return p, ops, rng.normal(0, 0.7, len(ops)), occ, oracle.Sector(n, na, nb)


# strings per spin: 84 x 84 (7,056), 70 x 56 (3,920: float-float), 252 x 120, 120 x 252, 55 x 462, 14 x 3,003 (49 columns), 210 x 210, 66 x 495
@pytest.mark.parametrize("n,na,nb", [(18, 3, 3), (16, 4, 3), (20, 5, 3), (20, 3, 5), (22, 2, 5), (28, 1, 6), (20, 4, 4), (24, 2, 4)])
def test_digit_products(n, na, nb):
    p, ops, theta, occ, sec = _problem(n, na, nb)
    Eref, gref = A.energy_grad(sec, p["h"], p["eri"], p["e_nuc"], ops, theta, A.hf_state(sec, occ))
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    got = {}
    for variant in (0, 3):
        st = sv.StateVector(n, "r64", sector=(na, nb))
        st.set_option(sv.SV_OPT_EXPECT_VARIANT, variant)
        st.prepare_hf(occ)
        for _ in range(2):
            got[variant] = st.energy_grad(ham, ops, theta)
            assert abs(got[variant][0] - Eref) <= TOL_E and np.max(np.abs(got[variant][1] - gref)) <= TOL_G
        st.close()
    # sums of 53 exact products against sums of thousands of rounded ones: a few hundred float64 steps
    assert np.max(np.abs(got[0][1] - got[3][1])) <= 1e-13 * max(1.0, np.max(np.abs(gref)))


@pytest.mark.parametrize("scale", [1e-120, 1e-3, 1e60])
def test_amplitude_scale(scale):
    """The digits stand under the largest amplitude's power of two: a state's scale drops out."""
    n, na, nb = 20, 4, 4
    p, ops, theta, occ, sec = _problem(n, na, nb)
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    dense = inputs.random_sector_state(n, na, nb, np.random.default_rng(4)).real
    dense /= np.linalg.norm(dense)
    E = []
    for s in (1.0, scale):
        st = sv.StateVector(n, "r64")
        st.prepare_state(dense * s, na, nb)
        E.append(st.energy(ham))
        st.close()
    assert abs(E[0] - A.energy(sec, p["h"], p["eri"], p["e_nuc"], dense[sec.dets.astype(np.int64)] + 0j)) <= TOL_E
    assert abs(E[1] - E[0]) <= TOL_E


def test_byte_caps_take_the_float_float_and_float64_sums():
    n, na, nb = 22, 4, 4
    p, ops, theta, occ, sec = _problem(n, na, nb)
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    E = []
    for cap in (0, 24 << 20, 6 << 20):
        st = sv.StateVector(n, "r64", sector=(na, nb))
        if cap:
            st.set_option(sv.SV_OPT_MAX_BYTES, cap)
        st.prepare_hf(occ)
        st.apply_ansatz(ops, theta)
        E.append(st.energy(ham))
        st.close()
    assert max(abs(E[1] - E[0]), abs(E[2] - E[0])) <= TOL_E


@pytest.mark.parametrize("stall", [1, 2, 3])
def test_bounded_wait_runs_out_reports_and_recovers(stall):
    n, na, nb = 20, 4, 4
    p, ops, theta, occ, sec = _problem(n, na, nb)
    Eref, _ = A.energy_grad(sec, p["h"], p["eri"], p["e_nuc"], ops, theta, A.hf_state(sec, occ))
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    st = sv.StateVector(n, "r64", sector=(na, nb))
    st.set_option(sv.SV_OPT_WAIT_POLLS, 4096)
    st.set_option(sv.SV_OPT_TEST_STALL, stall)
    st.prepare_hf(occ)
    with pytest.raises(sv.SvError) as e:
        st.energy_grad(ham, ops, theta)
    assert e.value.status == 3 and "bounded wait" in str(e.value)
    st.set_option(sv.SV_OPT_TEST_STALL, 0)
    st.set_option(sv.SV_OPT_WAIT_POLLS, 1 << 22)
    st.prepare_hf(occ)
    assert abs(st.energy_grad(ham, ops, theta)[0] - Eref) <= TOL_E
    st.close()


def test_float_float_can_be_chosen():
    """Variant 6 is the float-float form also where the automatic choice is the digit products: it has a sigma
    element of an amplitude 2^-44 of the largest, coupled to no other, to its own precision (48 bits a term).
    The gradient of the single excitation from that determinant at zero angle is that element alone."""
    n, na, nb = 20, 4, 4
    p = inputs.make_problem(n, 8, 4, seed=5)
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    bits = lambda orbs: sum((1 << 2 * q) | (1 << (2 * q + 1)) for q in orbs)  # noqa: E731
    psi = np.zeros(1 << n)
    psi[bits(range(4))] = 1.0
    psi[bits(range(6, 10))] = 0.7 * 2.0 ** -44      # eight excitations away
    op = np.array([(1, 12, -1, 10, -1)], np.int32)  # alpha, orbital 6 -> 5
    g = {}
    for variant in (0, 3, 6):
        st = sv.StateVector(n, "r64", sector=(na, nb))
        st.set_option(sv.SV_OPT_EXPECT_VARIANT, variant)
        st.prepare_state(psi, na, nb)
        g[variant] = st.energy_grad(ham, op, [0.0])[1][0]
        st.close()
    assert abs(g[3]) > 1e-30
    assert abs(g[6] - g[3]) <= 1e-12 * abs(g[3])     # some tens of terms of 2^-47
    assert abs(g[0] - g[3]) <= 2.0 ** -90            # an absolute 2^-52 of the largest, times the amplitude
    ham.close()
