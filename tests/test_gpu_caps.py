"""Device memory that runs short (SV_OPT_MAX_BYTES): whatever a handle keeps to be faster -- product planes,
sweep steps -- gives way, so a cap under which the plainest forms run is enough for every default call,
with the same results."""
import numpy as np
import pytest

from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu

# energy, gradient, 1-RDM: the parity suite's tolerances of each precision
TOL = {"c128": (1e-10, 1e-9, 1e-12), "r64": (1e-10, 1e-9, 1e-12), "c64": (1e-5, 1e-5, 2e-6), "r32": (1e-5, 1e-5, 2e-6)}
PLAIN = {sv.SV_OPT_EXPECT_VARIANT: 3, sv.SV_OPT_SECTOR_SWEEP: 0}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


def _problem(n, ne):
    p = inputs.make_problem(n, ne, 60, seed=n)
    return p, sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])


def _run(n, ne, dtype, cap, options, calls):
    """The results of calls(state) on a capped handle, None where one was refused for memory."""
    st = None
    try:
        st = sv.StateVector(n, dtype, sector=(ne // 2, ne // 2))
        st.set_option(sv.SV_OPT_MAX_BYTES, cap)
        for opt, value in options.items():
            st.set_option(opt, value)
        return calls(st)
    except sv.SvError as e:
        assert e.status == 2, e
        return None
    finally:
        if st is not None:
            st.close()


def _least_cap(run):
    """The least cap (to 2 KB) under which run(cap) is accepted."""
    lo, hi = 0, 256 << 20
    assert run(hi) is not None
    while hi - lo > 2048:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if run(mid) is not None else (mid, hi)
    return hi


def _check(got, want, tol, why):
    assert got is not None, ("refused", why)
    for (x, t), y in zip(got, want):
        assert np.max(np.abs(np.asarray(x) - np.asarray(y[0]))) <= tol[t], why


@pytest.mark.parametrize("dtype", ["r32", "c64"])
@pytest.mark.parametrize("n,ne", [(20, 10), (22, 8)])
def test_products_that_do_not_fit_leave_the_sparse_sums(n, ne, dtype):
    """63,504 and 108,900 determinants: the automatic choice is the tensor-core products."""
    p, ham = _problem(n, ne)

    def calls(st):
        st.prepare_hf(p["occ"])
        st.apply_ansatz(p["ops"], p["theta"])
        return [(st.energy(ham), 0)]

    plain = lambda cap: _run(n, ne, dtype, cap, PLAIN, calls)
    least = _least_cap(plain)
    want = plain(0)
    for factor in (1.0, 1.1, 1.5, 2.5, 6.0, 20.0):
        got = _run(n, ne, dtype, int(least * factor), {sv.SV_OPT_SECTOR_SWEEP: 0}, calls)
        _check(got, want, TOL[dtype], factor)
    ham.close()


@pytest.mark.parametrize("dtype", ["r32", "r64", "c128"])
@pytest.mark.parametrize("call", ["apply", "energy_grad"])
def test_sweep_steps_that_do_not_fit_leave_one_launch_per_operator(call, dtype):
    """A list of 600 operators over few determinants: the lists weigh more than the vectors."""
    p, ham = _problem(16, 4)
    pool = inputs.uccsd_pool(16, 4)
    ops = np.ascontiguousarray(pool[np.arange(600) % len(pool)])
    theta = np.random.default_rng(6).normal(0.0, 0.05, len(ops))

    def calls(st):
        st.prepare_hf(p["occ"])
        if call == "apply":
            st.apply_ansatz(ops, theta)
            return [(st.state(), 2)]
        E, g = st.energy_grad(ham, ops, theta)
        return [(E, 0), (g, 1), (st.state(), 2)]

    plain = lambda cap: _run(16, 4, dtype, cap, PLAIN, calls)
    least = _least_cap(plain)
    want = plain(0)
    for factor in (1.0, 1.02, 1.1, 1.3, 1.6, 2.0, 3.0):
        got = _run(16, 4, dtype, int(least * factor), {sv.SV_OPT_EXPECT_VARIANT: 3}, calls)
        _check(got, want, TOL[dtype], factor)
    ham.close()


@pytest.mark.parametrize("dtype", ["r64", "r32", "c64"])
def test_planes_give_way_to_later_calls(dtype):
    """The expectation may take what a cap leaves; the 1-RDM, the pool, a checkpointed sweep and a longer list
    after it are accepted wherever they are with the plain forms."""
    n, ne = 20, 8
    p, ham = _problem(n, ne)
    pool = inputs.uccsd_pool(n, ne)
    theta = np.random.default_rng(2).normal(0.0, 0.05, 400)

    def calls(st):
        st.prepare_hf(p["occ"])
        E, g = st.energy_grad(ham, p["ops"], p["theta"])
        out = [(E, 0), (g, 1), (st.rdm1(), 2)]
        E, g = st.energy_grad(ham, pool[:400], theta)
        out += [(E, 0), (g, 1), (st.rdm1(), 2)]
        E, g = st.pool_gradients(ham, pool)
        return out + [(E, 0), (g, 1)]

    plain = lambda cap: _run(n, ne, dtype, cap, PLAIN, calls)
    least = _least_cap(plain)
    want = plain(0)
    full = _run(n, ne, dtype, 0, {}, calls)
    _check(full, want, TOL[dtype], "no cap")
    for cap in range(least, 8 * least, max(least // 6, 1)):
        _check(_run(n, ne, dtype, cap, {}, calls), want, TOL[dtype], cap)
    ham.close()


def test_tables_that_do_not_fit_are_refused_again():
    """A dense handle whose string tables or compact matrix do not fit is refused each time it asks, not only
    the first, and serves a smaller sector in between."""
    n = 16
    p, ham = _problem(n, 8)
    big, small = p["occ"], p["occ"][:2]
    want = {}
    base = 8 << n
    for cap in [0] + list(range(base, base + 96 * 1024, 1536)):
        st = sv.StateVector(n, "c64")
        st.set_option(sv.SV_OPT_MAX_BYTES, cap)
        st.set_option(sv.SV_OPT_EXPECT_VARIANT, 3)
        for occ in (big, big, small, big, big, small):
            st.prepare_hf(occ)
            try:
                E = st.energy(ham)
            except sv.SvError as e:
                assert e.status == 2 and cap, e
                continue
            assert abs(E - want.setdefault(len(occ), E)) <= 1e-5, cap
        st.close()
    ham.close()
