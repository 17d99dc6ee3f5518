"""GPU parity of the batched persistent launch (config 4: 512 instances of 10-20
qubits, 40 operators each) against the CPU oracle, instance by instance."""
import numpy as np
import pytest

import oracle
from oracle import route_a as A
from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu

TOL = {"c128": (1e-10, 1e-9), "c64": (1e-5, 1e-5)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


def _oracle(p):
    sec = oracle.Sector(p["n_qubits"], p["na"], p["nb"])
    return A.energy_grad(sec, p["h"], p["eri"], p["e_nuc"], p["ops"], p["theta"], A.hf_state(sec, p["occ"]))


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_batch_matches_oracle_mixed_sizes(dtype):
    probs = inputs.batch_problems(24)
    assert len({p["n_qubits"] for p in probs}) >= 4
    b = sv.Batch(probs, dtype)
    theta = np.concatenate([p["theta"] for p in probs])
    E, g = b.energy_grad(theta)
    tE, tg = TOL[dtype]
    for k, p in enumerate(probs):
        Er, gr = _oracle(p)
        assert abs(E[k] - Er) <= tE, (k, p["n_qubits"], E[k], Er)
        assert np.max(np.abs(g[k] - gr)) <= tg, (k, p["n_qubits"])
    assert b.launches == 2  # the angles' cosines and sines, then the batched kernel


def test_batch_full_config4_sampled():
    """All 512 instances in one launch (complex64); instances of every size checked against the oracle."""
    probs = inputs.batch_problems(512)
    b = sv.Batch(probs, "c64")
    theta = np.concatenate([p["theta"] for p in probs])
    E, g = b.energy_grad(theta)
    assert np.all(np.isfinite(E))
    picked = {}
    for k, p in enumerate(probs):
        picked.setdefault(p["n_qubits"], []).append(k)
    for n, ks in sorted(picked.items()):
        for k in ks[:2]:
            Er, gr = _oracle(probs[k])
            assert abs(E[k] - Er) <= 1e-5, (n, k)
            assert np.max(np.abs(g[k] - gr)) <= 1e-5, (n, k)
    # a second launch with other angles gives other numbers, replayed from the same graph
    E2, _ = b.energy_grad(theta * 0.5)
    assert not np.allclose(E, E2)
    assert b.launches == 4


def test_batch_deterministic_and_same_as_single_handles():
    probs = inputs.batch_problems(10, first=100)
    b = sv.Batch(probs, "c128")
    theta = np.concatenate([p["theta"] for p in probs])
    E1, g1 = b.energy_grad(theta)
    E2, g2 = b.energy_grad(theta)
    assert np.array_equal(E1, E2) and all(np.array_equal(x, y) for x, y in zip(g1, g2))
    for k, p in enumerate(probs[:4]):
        ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
        st = sv.StateVector(p["n_qubits"], "c128")
        st.prepare_hf(p["occ"])
        E, g = st.energy_grad(ham, p["ops"], p["theta"])
        assert abs(E - E1[k]) <= 1e-11 and np.max(np.abs(g - g1[k])) <= 1e-10


def test_batch_time_limit_reports_timeout_and_recovers():
    probs = inputs.batch_problems(64)
    b = sv.Batch(probs, "c64")
    theta = np.concatenate([p["theta"] for p in probs])
    b.set_time_limit(1e-6)          # 1 ns: every block stops before taking a second instance
    with pytest.raises(sv.SvError) as e:
        b.energy_grad(theta)
    assert e.value.status == 4
    b.set_time_limit(0)
    E, g = b.energy_grad(theta)
    assert np.all(np.isfinite(E))


def test_batch_edges_and_errors():
    p = inputs.make_problem(8, 2, "uccsd", 5)
    empty = dict(p, ops=p["ops"][:0], theta=np.zeros(0))
    vac = dict(p, occ=[])
    b = sv.Batch([p, empty, vac], "c128")
    E, g = b.energy_grad(np.concatenate([p["theta"], [], p["theta"]]))
    Er, gr = _oracle(p)
    assert abs(E[0] - Er) <= 1e-10 and np.max(np.abs(g[0] - gr)) <= 1e-9
    sec = oracle.Sector(8, 1, 1)
    assert abs(E[1] - A.energy(sec, p["h"], p["eri"], p["e_nuc"], A.hf_state(sec, p["occ"]))) <= 1e-12
    assert len(g[1]) == 0
    assert abs(E[2] - p["e_nuc"]) <= 1e-12 and np.max(np.abs(g[2])) == 0.0
    bad = dict(p, ops=np.array([(2, 0, 1, 2, 2)], np.int32), theta=np.zeros(1))
    with pytest.raises(sv.SvError) as e:
        sv.Batch([bad], "c64")
    assert e.value.status == 1
    with pytest.raises(sv.SvError):
        b.energy_grad(np.full(2 * len(p["ops"]), np.nan))


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_batch_generic_path_for_large_string_spaces(dtype):
    """An instance with more than 512 alpha strings (24 qubits, 5 alpha + 1 beta electrons:
    792 x 12 determinants) takes the generic per-element sigma and filtered sweeps; batched
    beside instances that take the string-blocked path, every instance matches the oracle."""
    big = inputs.make_problem(24, 6, 12, seed=4242)
    big["occ"] = np.array([0, 2, 4, 6, 8, 1], dtype=np.int32)   # alpha orbitals 0-4, beta orbital 0
    big["na"], big["nb"] = 5, 1
    probs = [big] + inputs.batch_problems(3, first=7)
    b = sv.Batch(probs, dtype)
    theta = np.concatenate([p["theta"] for p in probs]) * 4
    E, g = b.energy_grad(theta)
    tE, tg = TOL[dtype]
    off = 0
    for k, p in enumerate(probs):
        q = dict(p, theta=theta[off:off + len(p["ops"])])
        off += len(p["ops"])
        Er, gr = _oracle(q)
        assert abs(E[k] - Er) <= tE, (k, E[k], Er)
        assert np.max(np.abs(g[k] - gr)) <= tg, k


@pytest.mark.parametrize("dtype,n,na,nb,n_ops", [("c128", 16, 2, 4, 20), ("c128", 18, 2, 2, 103), ("c64", 16, 2, 2, 217)])
def test_batch_shared_memory_just_below_48_kb(dtype, n, na, nb, n_ops):
    """Dynamic shared memory of 48,896, 48,448 and 48,336 bytes: below 48 KB, but with the kernel's own
    static part above the launch limit that holds until it is raised."""
    p = inputs.make_problem(n, 4, 4, seed=31)
    pool = inputs.uccsd_pool(n, 4)
    p["ops"] = np.ascontiguousarray(pool[np.arange(n_ops) % len(pool)])
    p["theta"] = np.random.default_rng(n_ops).normal(0.0, 0.05, n_ops)
    p["occ"] = [2 * k for k in range(na)] + [2 * k + 1 for k in range(nb)]
    p["na"], p["nb"] = na, nb
    b = sv.Batch([p, p], dtype)
    E, g = b.energy_grad(np.concatenate([p["theta"], p["theta"]]))
    Er, gr = _oracle(p)
    tE, tg = TOL[dtype]
    for k in range(2):
        assert abs(E[k] - Er) <= tE and np.max(np.abs(g[k] - gr)) <= tg
    b.close()


def _small(n, ne, n_ops, seed):
    p = inputs.make_problem(n, ne, 4, seed=seed)
    pool = inputs.uccsd_pool(n, ne)
    rng = np.random.default_rng(seed)
    p["ops"] = np.ascontiguousarray(pool[rng.integers(0, len(pool), n_ops)])
    p["theta"] = rng.normal(0.0, 0.2, n_ops)
    return p


def _check(probs, E, g, dtype, picked):
    tE, tg = TOL[dtype]
    for k in picked:
        Er, gr = _oracle(probs[k])
        assert abs(E[k] - Er) <= tE, (k, probs[k]["n_qubits"])
        assert np.max(np.abs(g[k] - gr), initial=0.0) <= tg, (k, probs[k]["n_qubits"])


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("count", [310, 620])
def test_batch_of_teams(count, big, dtype):
    """Small instances on half (310: at least two to an SM) and quarter blocks (620: four), alone and behind
    one that takes a whole block: every distinct problem against the oracle, copies of one bit for bit."""
    base = [_small(4, 2, 3, 1), _small(8, 2, 9, 2), _small(8, 4, 20, 3), _small(10, 4, 25, 4), _small(12, 4, 7, 5),
            dict(_small(12, 6, 30, 6)), _small(10, 4, 0, 7)]
    probs = ([_small(18, 6, 30, 8)] if big else []) + [base[k % len(base)] for k in range(count)]
    b = sv.Batch(probs, dtype)
    theta = np.concatenate([p["theta"] for p in probs])
    first = int(big)
    for again in range(2):
        E, g = b.energy_grad(theta)
        _check(probs, E, g, dtype, range(first + len(base)))
        for k in range(first, len(probs)):
            j = first + (k - first) % len(base)
            assert E[k] == E[j] and np.array_equal(g[k], g[j]), k
        if not again:
            b.autotune(theta)          # shared memory planned for one thread count, run with another
    b.close()


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,ne,n_ops", [(12, 6, 1500), (18, 6, 1200)])
def test_batch_lists_that_do_not_fit(n, ne, n_ops, dtype):
    """Operator lists longer than the shared memory beside the state: read from global memory; a batch of
    one, and one whose quarter blocks have little each."""
    p = _small(n, ne, n_ops, 40)
    for copies in (1, 610 if n == 12 else 2):
        b = sv.Batch([p] * copies, dtype)
        E, g = b.energy_grad(np.concatenate([p["theta"]] * copies))
        _check([p], E, g, dtype, [0])
        for k in range(1, copies):
            assert E[k] == E[0] and np.array_equal(g[k], g[0])
        b.close()
