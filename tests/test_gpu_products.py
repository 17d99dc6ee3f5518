"""The tensor-core products of single-precision states at the string counts where their tiles change width
(32, 64, 128 and 256 beta strings) and have ragged edges, against the float64 sums."""
import numpy as np
import pytest

from paper_2405_11567_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2405_11567_gb300 import build
    build.build()
    sv.lib()


# strings per spin and tile: below 2^20 determinants the alpha and the beta product in CTAs of their own, 330 x 165
# (five K blocks: two follow the small products) and 13 x 1,716 (a ragged edge on few rows) 32, 792 x 792 64 in two
# rounds; from there both in one, 3,003 x 364 64; 1,287 x 1,287 and 2,002 x 1,001 128 (complex: 256); 2,002 x 2,002 256
@pytest.mark.parametrize("dtype", ["r32", "c64"])
@pytest.mark.parametrize("n,na,nb", [(22, 4, 3), (26, 1, 6), (24, 5, 5), (28, 6, 3), (26, 5, 5), (28, 4, 5), (28, 5, 5)])
def test_products_at_every_tile_width(n, na, nb, dtype):
    rng = np.random.default_rng(n + nb)
    p = inputs.make_problem(n, 8, 4, seed=n)
    pool = inputs.qeb_pool(n, 8)
    ops = pool[rng.integers(0, len(pool), 12)]
    theta = rng.normal(0, 0.3, len(ops))
    occ = [2 * k for k in range(na)] + [2 * k + 1 for k in range(nb)]
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    out = {}
    for dt, variant in (("r64", 3), (dtype, 4), (dtype, 5)):
        st = sv.StateVector(n, dt, sector=(na, nb))
        st.set_option(sv.SV_OPT_EXPECT_VARIANT, variant)
        st.set_option(sv.SV_OPT_FULL_VECTOR, 1)      # complex planes for complex64
        st.prepare_hf(occ)
        out[dt, variant] = st.energy_grad(ham, ops, theta)
        st.close()
    E, g = out["r64", 3]
    for variant in (4, 5):
        assert abs(out[dtype, variant][0] - E) <= 1e-5          # the parity suite's complex64 tolerances
        assert np.max(np.abs(out[dtype, variant][1] - g)) <= 1e-5
    ham.close()
