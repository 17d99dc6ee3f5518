"""The compute core (dense handles on their sector's amplitudes, complex handles with a real
reference in real amplitudes) against the full-vector route (SV_OPT_FULL_VECTOR = 1) and the
oracle: every call of the path, both storages, every type, determinants and stored real and
complex references, in every order that moves the state between the two."""
import ctypes

import numpy as np
import pytest

import oracle
from oracle import route_a as A
from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu

# energy, gradient, amplitudes and 1-RDM: the parity suite's tolerances of each precision
TOL = {"c128": (1e-10, 1e-9, 1e-12, 1e-12), "c64": (1e-5, 1e-5, 2e-6, 2e-6)}
NP = {"c128": np.complex128, "c64": np.complex64, "r64": np.float64, "r32": np.float32}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


def _start(start, n, na, nb, rng):
    dense = np.zeros(1 << n, dtype=np.complex128)
    if start == "hf":
        dense[sum(1 << j for j in _occ(na, nb))] = 1.0
    else:
        dense = inputs.random_sector_state(n, na, nb, rng)
        if start == "real":
            dense = dense.real / np.linalg.norm(dense.real) + 0j
    return dense


def _occ(na, nb):
    return [2 * p for p in range(na)] + [2 * p + 1 for p in range(nb)]


@pytest.mark.parametrize("storage", ["dense", "sector"])
@pytest.mark.parametrize("dtype", ["c128", "c64", "r64", "r32"])
@pytest.mark.parametrize("start", ["hf", "real", "complex"])
@pytest.mark.parametrize("na,nb", [(3, 2), (1, 4), (5, 5), (0, 1)])
def test_core_matches_full_vector_and_oracle(na, nb, start, dtype, storage):
    if start == "complex" and dtype.startswith("r"):
        pytest.skip("a real handle takes real states")
    n = 10
    rng = np.random.default_rng(10 * na + nb)
    p = inputs.make_problem(n, 4, 20, seed=77 + na)
    ops = np.vstack([p["ops"], inputs.qeb_pool(n, 4)[::9]])
    theta = rng.normal(0, 0.3, len(ops))
    dense0 = _start(start, n, na, nb, rng)
    sec = oracle.Sector(n, na, nb)
    at = sec.dets.astype(np.int64)
    psi0 = np.ascontiguousarray(dense0[at])
    Eref, gref = A.energy_grad(sec, p["h"], p["eri"], p["e_nuc"], ops, theta, psi0)
    psi = A.apply_ansatz(sec, ops, theta, psi0)
    rdm = A.rdm1(sec, psi)
    sig = A.hamiltonian_apply(sec, p["h"], p["eri"], p["e_nuc"], psi)
    pool = inputs.uccsd_pool(n, 4)
    gpool = np.array([2 * np.vdot(sig, A.generator_apply(sec, op, psi)).real for op in pool])
    tE, tg, ta, tr = TOL["c128" if dtype in ("c128", "r64") else "c64"]
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])

    def prepare(st):
        if start == "hf":
            st.prepare_hf(_occ(na, nb))
        else:
            st.prepare_state((dense0 if dtype.startswith("c") else dense0.real).astype(NP[dtype]), na, nb)

    def check_state(st, want, why):
        got = st.state()
        assert np.max(np.abs(got[at] - want)) <= ta, why
        assert np.count_nonzero(np.delete(got, at)) == 0, why
        assert np.array_equal(st.amplitudes(at[::3]), got[at[::3]]), why

    for full in (0, 1):
        st = sv.StateVector(n, dtype, sector=(na, nb) if storage == "sector" else None)
        st.set_option(sv.SV_OPT_FULL_VECTOR, full)
        prepare(st)
        check_state(st, psi0, "reference")
        assert abs(st.energy(ham) - A.energy(sec, p["h"], p["eri"], p["e_nuc"], psi0)) <= tE
        for _ in range(2):                                   # the second call on kept buffers
            E, g = st.energy_grad(ham, ops, theta)
            assert abs(E - Eref) <= tE and np.max(np.abs(g - gref)) <= tg, full
            check_state(st, psi, "after energy_grad")
            assert np.max(np.abs(st.rdm1() - rdm)) <= tr
        prepare(st)
        st.apply_ansatz(ops[:7], theta[:7])                  # in two parts: the state moves on
        st.apply_ansatz(ops[7:], theta[7:])
        check_state(st, psi, "after apply_ansatz")
        Ep, gp = st.pool_gradients(ham, pool)
        assert abs(Ep - Eref) <= tE and np.max(np.abs(gp - gpool)) <= tg
        st.set_option(sv.SV_OPT_FULL_VECTOR, 1 - full)       # the other route takes the state over
        assert abs(st.energy(ham) - Eref) <= tE
        st.apply_ansatz(ops[::-1], -theta[::-1])             # back to the reference
        check_state(st, psi0, "uncomputed")
        if storage == "dense":
            st.set_layout(rng.permutation(n))                # moves psi; the state is the same
            check_state(st, psi0, "moved")
            st.apply_ansatz(ops, theta)
            check_state(st, psi, "in another layout")
        E, g = st.energy_grad(ham, ops, theta)
        assert abs(E - Eref) <= tE and np.max(np.abs(g - gref)) <= tg
        check_state(st, psi, "energy_grad in another layout")
        st.close()


@pytest.mark.parametrize("storage", ["dense", "sector"])
def test_a_written_state_is_read_from_its_vector(storage):
    """Once the address is known outside, the caller may write there: energy, 1-RDM, ansatz and
    pool gradients take the amplitudes that are there, imaginary parts included; energy_grad
    starts from the reference and writes the whole vector, zeros outside the sector too."""
    n, na, nb = 10, 2, 2
    p = inputs.make_problem(n, 4, 15, seed=5)
    sec = oracle.Sector(n, na, nb)
    at = sec.dets.astype(np.int64)
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    want = inputs.random_sector_state(n, na, nb, np.random.default_rng(8))
    src = sv.StateVector(n, "c128", sector=(na, nb) if storage == "sector" else None)
    src.prepare_state(want, na, nb)
    st = sv.StateVector(n, "c128", sector=(na, nb) if storage == "sector" else None)
    st.set_option(sv.SV_OPT_LAYOUT_AUTO, 0)
    st.prepare_hf(p["occ"])
    Eref, gref = st.energy_grad(ham, p["ops"], p["theta"])
    psi = st.state()

    def write():
        size = 16 * (sec.D if storage == "sector" else 1 << n)
        a, b = sv.sv_state_device_ptr(st.handle), sv.sv_state_device_ptr(src.handle)
        rt = ctypes.CDLL("libcudart.so.13")
        assert rt.cudaDeviceSynchronize() == 0
        assert rt.cudaMemcpy(ctypes.c_void_p(a), ctypes.c_void_p(b), ctypes.c_size_t(size), 3) == 0  # device to device

    write()
    E = A.energy(sec, p["h"], p["eri"], p["e_nuc"], want[at])
    assert abs(st.energy(ham) - E) <= 1e-10
    assert np.max(np.abs(st.rdm1() - A.rdm1(sec, want[at]))) <= 1e-12
    st.apply_ansatz(p["ops"], p["theta"])
    assert np.max(np.abs(st.state()[at] - A.apply_ansatz(sec, p["ops"], p["theta"], want[at]))) <= 1e-12
    E2, g2 = st.energy_grad(ham, p["ops"], p["theta"])
    assert abs(E2 - Eref) <= 1e-12 and np.max(np.abs(g2 - gref)) <= 1e-11
    assert np.max(np.abs(st.state() - psi)) <= 1e-13


def _overlapping_ops(n):
    """Every ordered pair of operators that share flip-mask bits in every way: disjoint, one
    orbital shared, the same masks with other "from" patterns, a single inside a double."""
    base = [(1, 0, -1, 4, -1), (1, 4, -1, 0, -1), (1, 1, -1, 5, -1), (1, 2, -1, 6, -1), (2, 0, 1, 4, 5), (2, 0, 5, 1, 4),
            (2, 0, 2, 4, 6), (2, 2, 3, 6, 7), (2, 0, 3, 4, 7), (2, 1, 3, 5, 7), (4, 0, 1, 4, 7), (3, 2, -1, 4, -1)]
    base = [op for op in base if max(op[1:]) < n]
    return np.array([op for a in base for b in base for op in (a, b)], np.int32)


@pytest.mark.parametrize("dtype", ["c128", "c64", "r64", "r32"])
@pytest.mark.parametrize("n,na,nb", [(8, 2, 2), (10, 3, 2), (16, 4, 4), (22, 5, 4)])
def test_paired_steps_match_single_operators(n, na, nb, dtype):
    """Whole sweeps, two operators to a step, in the block (8, 10 qubits), the cluster (16) and
    the grid form (22), against one launch per operator (SV_OPT_SECTOR_SWEEP = 0), for every way
    in which a step's two masks can overlap, an odd number of operators and operators without a
    pair: the same states and gradients, within the rounding of each pair's rotation, whose
    operands are the same."""
    rng = np.random.default_rng(n)
    ops = _overlapping_ops(n)
    if n > 16:
        ops = ops[:61]
    elif n == 16:
        ops = np.vstack([inputs.adapt_list(inputs.uccsd_pool(n, 8), 40, rng), ops[:101]])
    theta = rng.normal(0, 0.4, len(ops))
    theta[3] = 2.0                                       # cos < 0: not three shears
    h, eri, e_nuc = inputs.synthetic_integrals(n // 2, rng)
    ham = sv.Hamiltonian(h, eri, e_nuc)
    dense = inputs.random_sector_state(n, na, nb, rng)
    if dtype.startswith("r"):
        dense = dense.real / np.linalg.norm(dense.real)
    out = []
    for mode, polls in ((0, 1 << 22), (1, 1 << 22), (1, 1000)):    # 1000 polls: the grid form at every size
        st = sv.StateVector(n, dtype, sector=(na, nb))
        st.set_option(sv.SV_OPT_SECTOR_SWEEP, mode)
        st.set_option(sv.SV_OPT_WAIT_POLLS, polls)
        st.prepare_state(dense.astype(NP[dtype]), na, nb)
        E, g = st.energy_grad(ham, ops, theta)
        out.append((E, g, st.state()))
        st.close()
    eps = 2.3e-16 if dtype in ("c128", "r64") else 1.2e-7
    scale = np.max(np.abs(out[0][1])) + 1.0
    for E, g, psi in out[1:]:
        assert np.max(np.abs(psi - out[0][2])) <= 4 * len(ops) * eps
        assert abs(E - out[0][0]) <= 64 * len(ops) * eps
        assert np.max(np.abs(g - out[0][1])) <= 64 * len(ops) * eps * scale


@pytest.mark.parametrize("dtype", ["c128", "c64", "r64", "r32"])
def test_prepare_again_leaves_one_amplitude(dtype):
    """A determinant prepared over an earlier state of the same sector (few of the vector's amplitudes),
    of another sector, in a moved layout and after whole-vector calls: one amplitude, and its energy."""
    n = 16
    p = inputs.make_problem(n, 4, 20, seed=12)
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    rng = np.random.default_rng(3)
    st = sv.StateVector(n, dtype)
    occs = [_occ(2, 2), _occ(2, 2), [0, 4, 3, 9], _occ(1, 2), _occ(2, 2), _occ(2, 2)]
    for k, occ in enumerate(occs):
        st.prepare_hf(occ)
        if k == 3:
            st.set_option(sv.SV_OPT_FULL_VECTOR, 1)
        if k == 4:
            st.set_option(sv.SV_OPT_FULL_VECTOR, 0)
        st.energy_grad(ham, p["ops"], p["theta"])
        if k == 1:
            st.set_layout(rng.permutation(n))
        st.prepare_hf(occ)
        got = st.state()
        x = sum(1 << j for j in occ)
        assert np.count_nonzero(got) == 1 and got[x] == 1.0, k
        sec = oracle.Sector(n, sum(j % 2 == 0 for j in occ), sum(j % 2 for j in occ))
        assert abs(st.energy(ham) - A.energy(sec, p["h"], p["eri"], p["e_nuc"], A.hf_state(sec, occ))) <= TOL[
            {"r64": "c128", "r32": "c64"}.get(dtype, dtype)][0]
        st.apply_ansatz(p["ops"], p["theta"])
    st.close()
