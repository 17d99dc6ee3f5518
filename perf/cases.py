"""The work this framework does for its users, as cases that can be measured.

A case is one call, or the few calls that belong together, of a program that runs VQE or
ADAPT-VQE on the state-vector emulator, with everything such a program keeps between its
iterations (the handle, the Hamiltonian, the operator list) prepared before:

  energy    the HF state, the ansatz, <H> and the whole state read back (an optimiser
            without gradients; small registers)
  gradient  energy and gradient through ``autograd.energy`` (a torch optimiser)
  step      energy, adjoint gradient and 1-RDM, and the amplitudes of the reference and of
            the determinants its pool excites (one iteration of VQE with the density-based
            correction, with the leading coefficients that a user looks at)
  screen    the HF state, the current ansatz and the gradients of every pool operator (the
            selection step of ADAPT-VQE)
  batch     energies and gradients of many small problems in one launch

Problems come from ``inputs``: synthetic integrals with the shapes of the paper's
molecules, its operator pools and angles.  Sizes are those of the workloads there
(8, 16, 24 and 30 qubits, 512 batched instances of 10 to 20), and odd ones between.

A single-precision state gives single-precision numbers: the library accumulates and
returns its sums in float64, but they carry the rounding of the float32 amplitudes, so the
cases hand them on as float32, the type of what was computed.
"""
import functools

import numpy as np
import torch

from paper_2405_11567_gb300 import autograd, inputs, sv

SINGLE = ("c64", "r32")


def _case(kind, n_qubits, n_elec, n_ops, dtype, storage, pool="uccsd", start="hf", count=1):
    """n_ops: operators of the ansatz (0: the whole pool in order); count: batched instances;
    a batch's n_qubits is that of its largest instances (n_elec, pool and start don't apply)."""
    return dict(kind=kind, n_qubits=n_qubits, n_elec=n_elec, n_ops=n_ops, dtype=dtype, storage=storage, pool=pool,
                start=start, count=count)


def listed():
    return [
        # two electrons in four orbitals, UCCSD: the smallest molecule, where launches and latency count
        dict(_case("energy", 8, 2, 0, "c128", "dense"), name="energy_8q_c128"),
        # UCCSD with all its singles and doubles, driven by a torch optimiser
        dict(_case("gradient", 16, 4, 0, "c128", "dense"), name="gradient_16q_c128"),
        # the continuation of an ADAPT run from a multi-determinant state (any complex state may be given)
        dict(_case("step", 20, 8, 90, "c128", "dense", start="multi"), name="step_20q_multi_c128"),
        # an open shell, five alpha and four beta electrons in eleven orbitals, in real amplitudes
        dict(_case("step", 22, 9, 75, "r64", "sector"), name="step_22q_open_r64"),
        # a mid-sized ADAPT ansatz, in both precisions
        dict(_case("step", 24, 8, 120, "c64", "dense"), name="step_24q_c64"),
        dict(_case("step", 24, 8, 120, "c128", "dense"), name="step_24q_c128"),
        # the paper's operator selection, from its qubit-excitation pool
        dict(_case("screen", 28, 10, 60, "c64", "sector", pool="qeb"), name="screen_28q_qeb_c64"),
        # many small molecules or geometries at once
        dict(_case("batch", 20, 0, 40, "c64", "sector", count=512), name="batch_512_c64"),
        dict(_case("batch", 16, 0, 25, "c128", "sector", count=37), name="batch_37_c128"),
        # the largest ansatz of the workload list, in both storages and both precisions
        dict(_case("step", 30, 10, 200, "c64", "sector"), name="step_30q_sector_c64"),
        dict(_case("step", 30, 10, 200, "c64", "dense"), name="step_30q_c64"),
        dict(_case("step", 30, 10, 200, "c128", "dense"), name="step_30q_c128"),
    ]


def _between(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return min(hi, int(round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    kind = rng.choice(("energy", "gradient", "step", "step", "step", "screen", "batch"))
    if kind == "batch":
        n = 2 * rng.randint(5, 10)
        dtype = rng.choice(("c64", "c128"))
        return _case(kind, n, 0, _between(rng, 5, 40), dtype, "sector", count=_between(rng, 5, 512))
    n = 2 * rng.randint(*{"energy": (4, 6), "gradient": (5, 10)}.get(kind, (6, 14)))
    n_elec = rng.randint(2, min(n // 2 + 1, 12))
    dtype = rng.choice(("c64", "c64", "c128", "c128", "r32", "r64"))
    storage = rng.choice(("dense", "sector"))
    pool = rng.choice(("uccsd", "uccsd", "qeb"))
    start = rng.choice(("hf", "hf", "hf", "multi")) if kind == "step" and n <= 22 else "hf"
    return _case(kind, n, n_elec, _between(rng, 8, 200), dtype, storage, pool=pool, start=start)


# ---------------------------------------------------------------- inputs


def _sector(n_elec):
    return (n_elec + 1) // 2, n_elec // 2


def _problem(case, seed):
    p = inputs.make_problem(case["n_qubits"], case["n_elec"], case["n_ops"] or "uccsd", seed)
    if case["pool"] == "qeb":
        p["ops"][:, 0] += 2
    p["na"], p["nb"] = _sector(case["n_elec"])
    return p


def _batch_problems(case, seed):
    rng = np.random.default_rng(seed)
    smallest = 10 if case["n_qubits"] >= 18 else 8
    qubits = rng.choice(np.arange(smallest, case["n_qubits"] + 1, 2), size=case["count"])
    qubits[0] = case["n_qubits"]
    seeds = rng.integers(1 << 30, size=case["count"])
    sizes = [(int(q), inputs.batch_electrons(q)) for q in qubits]
    return [inputs.make_problem(*size, case["n_ops"], int(k)) for size, k in zip(sizes, seeds)]


def _pool(case):
    return (inputs.qeb_pool if case["pool"] == "qeb" else inputs.uccsd_pool)(case["n_qubits"], case["n_elec"])


def _determinants(case):
    """The reference and the determinants that the pool's operators excite it to."""
    ref = (1 << case["n_elec"]) - 1
    ops = inputs.uccsd_pool(case["n_qubits"], case["n_elec"])
    bits = np.where(ops[:, 1:] >= 0, np.uint64(1) << np.maximum(ops[:, 1:], 0).astype(np.uint64), np.uint64(0))
    return np.concatenate([[np.uint64(ref)], np.uint64(ref) ^ np.bitwise_or.reduce(bits, axis=1)]).astype(np.uint64)


def _start_state(case, seed):
    """A few hundred leading determinants with decaying weights (complex unless the state is real)."""
    rng = np.random.default_rng(seed + 1)
    x = _determinants(case)[:300].astype(np.int64)
    v = rng.normal(size=len(x)) * 0.1
    if case["dtype"].startswith("c"):
        v = v + 1j * rng.normal(size=len(x)) * 0.1
    v[0] = 1.0
    out = np.zeros(1 << case["n_qubits"], dtype=v.dtype)
    out[x] = v / np.linalg.norm(v)
    return out


# ---------------------------------------------------------------- the measured calls


def prepare(case, seed):
    if case["kind"] == "batch":
        problems = _batch_problems(case, seed)
        theta = np.concatenate([p["theta"] for p in problems])
        return dict(case=case, batch=sv.Batch(problems, case["dtype"]), theta=theta)
    p = _problem(case, seed)
    sector = (p["na"], p["nb"]) if case["storage"] == "sector" else None
    st = sv.StateVector(case["n_qubits"], case["dtype"], sector=sector)
    if case["start"] == "multi":
        st.prepare_state(_start_state(case, seed), p["na"], p["nb"])
    else:
        st.prepare_hf(p["occ"])
    ham = sv.Hamiltonian(p["h"], p["eri"], p["e_nuc"])
    s = dict(case=case, st=st, ham=ham, occ=p["occ"], ops=p["ops"], theta=p["theta"])
    if case["kind"] == "screen":
        s["pool"] = _pool(case)
    if case["kind"] == "step":
        s["dets"] = _determinants(case)
    return s


def _as_computed(case, out):
    """The numbers of a single-precision state in single precision."""
    if case["dtype"] not in SINGLE:
        return out
    return {k: np.asarray(v).astype(np.complex64 if np.iscomplexobj(v) else np.float32) for k, v in out.items()}


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        E, g = s["batch"].energy_grad(s["theta"])
        return _as_computed(case, dict(energy=E, gradient=np.concatenate(g)))
    st, ham = s["st"], s["ham"]
    if case["kind"] == "energy":
        st.prepare_hf(s["occ"])
        st.apply_ansatz(s["ops"], s["theta"])
        return _as_computed(case, dict(energy=st.energy(ham), state=st.state()))
    if case["kind"] == "gradient":
        theta = torch.from_numpy(s["theta"]).clone().requires_grad_()
        E = autograd.energy(theta, st, ham, s["ops"])
        E.backward()
        return _as_computed(case, dict(energy=E.item(), gradient=theta.grad.numpy()))
    if case["kind"] == "screen":
        st.prepare_hf(s["occ"])
        st.apply_ansatz(s["ops"], s["theta"])
        E, g = st.pool_gradients(ham, s["pool"])
        return _as_computed(case, dict(energy=E, gradient=g))
    E, g = st.energy_grad(ham, s["ops"], s["theta"])
    return _as_computed(case, dict(energy=E, gradient=g, rdm=st.rdm1(), amplitudes=st.amplitudes(s["dets"])))


# ---------------------------------------------------------------- what a pass cannot do without


def _choose(n, k):
    return 0 if k < 0 or k > n else functools.reduce(lambda r, i: r * (n - i) // (i + 1), range(k), 1)


def _one(n_qubits, n_elec, ops, kind, n_pool=0, cx=1):
    """(flops, bytes of inputs and of numbers returned) of one problem in the sector of its
    electrons; cx: numbers per amplitude (1 where the state is real: real angles and a real start)."""
    N, (na, nb) = n_qubits // 2, _sector(n_elec)
    D = _choose(N, na) * _choose(N, nb)
    sa, sb = na * (N - na), nb * (N - nb)
    links = 1 + sa + sb + sa * sb + _choose(na, 2) * _choose(N - na, 2) + _choose(nb, 2) * _choose(N - nb, 2)

    def pairs(op):  # determinants that the operator's "from" pattern matches
        occ, vir = [j for j in op[1:3] if j >= 0], [j for j in op[3:5] if j >= 0]
        n = 1
        for s, ne in ((0, na), (1, nb)):
            o, v = sum(j % 2 == s for j in occ), sum(j % 2 == s for j in vir)
            n *= _choose(N - o - v, ne - o)
        return n

    rotated = sum(pairs(op) for op in ops.tolist())
    flops = 2.0 * cx * D * links + 6.0 * cx * rotated * (1 if kind in ("energy", "screen") else 4)
    if kind == "step":
        flops += 2.0 * cx * D * (1 + N * N)
    flops += 4.0 * cx * n_pool * D / 16
    return flops, 8.0 * (N**4 + N**2 + 3 * len(ops) + 2 + 2 * n_pool)


def work(case):
    if case["kind"] == "batch":
        each = [_one(p["n_qubits"], p["n_elec"], p["ops"], "gradient") for p in _batch_problems(case, 1)]
        return dict(bytes=sum(b for _, b in each), flops=sum(f for f, _ in each))
    pool = _pool(case)
    ops = inputs.adapt_list(pool, case["n_ops"], np.random.default_rng(1)) if case["n_ops"] else pool
    n_pool = len(pool) if case["kind"] == "screen" else 0
    cx = 2 if case["start"] == "multi" and case["dtype"].startswith("c") else 1
    flops, nbytes = _one(case["n_qubits"], case["n_elec"], ops, case["kind"], n_pool, cx)
    # psi(theta), which the handle holds afterwards, in its storage
    na, nb = _sector(case["n_elec"])
    N = case["n_qubits"] // 2
    amplitude = {"c64": 8, "c128": 16, "r32": 4, "r64": 8}[case["dtype"]]
    held = 1 << case["n_qubits"] if case["storage"] == "dense" else _choose(N, na) * _choose(N, nb)
    if case["kind"] == "step":
        nbytes += 8.0 * 4 * N * N + amplitude * len(pool)
    return dict(bytes=nbytes + float(amplitude) * held, flops=flops)


# ---------------------------------------------------------------- the same in 64 bits, with torch


def _parity(x):
    for s in (16, 8, 4, 2, 1):
        x = x ^ (x >> s)
    return x & 1


class _Sector:
    """Amplitudes of one (na, nb) sector as a matrix [beta string][alpha string], spin-orbital
    j = 2p + spin at bit j of a determinant, Jordan-Wigner order."""

    def __init__(self, N, na, nb, device):
        self.N = N
        words = torch.arange(1 << N, device=device)
        ones = sum((words >> p) & 1 for p in range(N))
        self.strings = [words[ones == k] for k in (na, nb)]
        self.rank, self.spread = [], []
        for spin, s in enumerate(self.strings):
            rank = torch.full((1 << N,), -1, device=device)
            rank[s] = torch.arange(len(s), device=device)
            self.rank.append(rank)
            self.spread.append(sum(((s >> p) & 1) << (2 * p + spin) for p in range(N)))
        self.shape = (len(self.strings[1]), len(self.strings[0]))
        self.known = {}

    def index(self, x):
        """The flat positions of the determinants x (a numpy array)."""
        one, at = np.uint64(1), []
        for spin, rank in enumerate(self.rank):
            s = sum(((x >> np.uint64(2 * p + spin)) & one) << np.uint64(p) for p in range(self.N))
            at.append(rank[torch.from_numpy(s.astype(np.int64)).to(rank.device)])
        return at[1] * self.shape[1] + at[0]

    def excitation(self, op):
        """T of the operator row as (from, to, sign): flat positions and the sign of each pair."""
        key = tuple(int(v) for v in op)
        if key in self.known:
            return self.known[key]
        kind, i, j, a, b = key
        occ, vir = ([i], [a]) if kind in (1, 3) else ([i, j], [a, b])
        moved = []
        for spin in (0, 1):
            f = sum(1 << (q // 2) for q in occ if q % 2 == spin)
            t = sum(1 << (q // 2) for q in vir if q % 2 == spin)
            s = self.strings[spin]
            at = torch.nonzero((s & (f | t)) == f).reshape(-1)
            moved.append((at, self.rank[spin][s[at] ^ (f | t)], self.spread[spin][at]))
        (ca, ta, xa), (cb, tb, xb) = moved
        src, dst = cb[:, None] * self.shape[1] + ca, tb[:, None] * self.shape[1] + ta
        sign = torch.ones(src.shape, dtype=torch.float64, device=src.device)
        if kind in (1, 2):  # a+_a (a+_b a_j) a_i, rightmost first, each counting the occupied orbitals below it
            odd = torch.zeros(src.shape, dtype=torch.int64, device=src.device)
            done = 0
            for q in occ + vir[::-1]:
                low = (1 << q) - 1
                odd ^= (_parity(xa & low) ^ (bin(done & low).count("1") & 1)) ^ _parity(xb & low)[:, None]
                done ^= 1 << q
                sign = 1.0 - 2.0 * odd.to(torch.float64)
        got = (src.reshape(-1), dst.reshape(-1), sign.reshape(-1))
        if len(got[0]) < 100_000:
            self.known[key] = got
        return got

    def rotate(self, op, theta, *vectors):
        src, dst, sign = self.excitation(op)
        c, s = float(np.cos(theta)), float(np.sin(theta)) * sign
        for v in vectors:
            u, w = v[src], v[dst]
            v[src], v[dst] = c * u - s * w, c * w + s * u

    def generator(self, op, left, right):
        """Re <left| T - T^dagger |right>"""
        src, dst, sign = self.excitation(op)
        return float((sign * (left[dst].conj() * right[src] - left[src].conj() * right[dst]).real).sum())

    def _moves(self, spin, p, q):
        """a+_p a_q of one spin on strings: (from, to, sign by the alpha string, sign by the beta string)."""
        key = ("move", spin, p, q)
        if key not in self.known:
            s = self.strings[spin]
            at = torch.nonzero(((s >> q) & 1 == 1) & (((s >> p) & 1 == 0) | (p == q))).reshape(-1)
            to = self.rank[spin][(s[at] ^ (1 << q)) | (1 << p)]
            lo, hi = sorted((2 * p + spin, 2 * q + spin))
            mask = ((1 << hi) - 1) & ~((1 << (lo + 1)) - 1)
            signs = [1.0 - 2.0 * _parity(x & mask).to(torch.float64) for x in self.spread]
            signs[spin] = signs[spin][at]
            self.known[key] = (at, to, signs[0], signs[1])
        return self.known[key]

    def one_body(self, spin, p, q, C):
        """a+_p a_q of one spin, on the matrix C."""
        at, to, sa, sb = self._moves(spin, p, q)
        out = torch.zeros_like(C)
        if spin == 0:
            out[:, to] = C[:, at] * sa * sb[:, None]
        else:
            out[to] = C[at] * sb[:, None] * sa
        return out

    def hamiltonian(self, h, eri, e_nuc, v):
        """H v, with H = sum k_pq E_pq + 1/2 sum (pq|rs) E_pq E_rs + e_nuc over spin-summed E,
        k_pq = h_pq - 1/2 sum_r (pr|rq)."""
        C, N = v.reshape(self.shape), self.N
        pairs = [(p, q) for p in range(N) for q in range(p + 1)]

        def both(p, q, X):
            y = self.one_body(0, p, q, X) + self.one_body(1, p, q, X)
            return y if p == q else y + self.one_body(0, q, p, X) + self.one_body(1, q, p, X)

        D = torch.stack([both(p, q, C) for p, q in pairs])
        k = h - 0.5 * np.einsum("prrq->pq", eri)
        p, q = (np.array(t) for t in zip(*pairs))
        W = torch.from_numpy(0.5 * eri[p[:, None], q[:, None], p, q]).to(C.device)
        kt = torch.from_numpy(k[p, q]).to(C.device)
        flat = torch.view_as_real(D).reshape(len(pairs), -1) if D.is_complex() else D.reshape(len(pairs), -1)

        def matrix(row):
            return torch.view_as_complex(row.reshape(*C.shape, 2)) if D.is_complex() else row.reshape(C.shape)

        out, G = e_nuc * C + matrix(kt @ flat), W @ flat
        for (a, b), g in zip(pairs, G):
            out += both(a, b, matrix(g))
        return out.reshape(-1)

    def rdm(self, v):
        C, N = v.reshape(self.shape), self.N
        out = np.zeros((2, N, N), dtype=np.complex128)
        for spin in (0, 1):
            for p in range(N):
                for q in range(p, N):
                    out[spin, p, q] = complex((C.conj() * self.one_body(spin, p, q, C)).sum())
                    out[spin, q, p] = out[spin, p, q].conjugate()
        return out / float((v.conj() * v).real.sum())


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _forward(sec, p, start):
    psi = start.clone()
    for op, t in zip(p["ops"], p["theta"]):
        sec.rotate(op, t, psi)
    return psi


def _energy_gradient(sec, p, psi):
    """E and dE/dtheta at psi = psi(theta)."""
    lam = sec.hamiltonian(p["h"], p["eri"], p["e_nuc"], psi)
    norm = float((psi.conj() * psi).real.sum())
    E = float((psi.conj() * lam).real.sum()) / norm
    psi, g = psi.clone(), np.zeros(len(p["ops"]))
    for k in range(len(g) - 1, -1, -1):
        g[k] = 2.0 * sec.generator(p["ops"][k], lam, psi) / norm
        sec.rotate(p["ops"][k], -p["theta"][k], psi, lam)
    return E, g


def _reference(sec, p):
    psi = torch.zeros(sec.shape[0] * sec.shape[1], dtype=torch.float64, device=_device())
    psi[sec.index(np.array([(1 << p["n_elec"]) - 1], dtype=np.uint64))] = 1.0
    return psi


def exact(case, seed):
    if case["kind"] == "batch":
        problems, secs, E, g = _batch_problems(case, seed), {}, [], []
        for p in problems:
            key = (p["n_orb"], p["na"], p["nb"])
            if key not in secs:
                secs[key] = _Sector(*key, _device())
            sec = secs[key]
            e, gr = _energy_gradient(sec, p, _forward(sec, p, _reference(sec, p)))
            E.append(e)
            g.append(gr)
        return dict(energy=np.array(E), gradient=np.concatenate(g))
    p = _problem(case, seed)
    sec = _Sector(p["n_orb"], p["na"], p["nb"], _device())
    if case["start"] == "multi":
        v, x = _start_state(case, seed), _determinants(case)[:300]
        start = torch.zeros(sec.shape[0] * sec.shape[1], dtype=torch.from_numpy(v).dtype, device=_device())
        start[sec.index(x)] = torch.from_numpy(v[x.astype(np.int64)]).to(_device())
    else:
        start = _reference(sec, p)
    psi = _forward(sec, p, start)
    if case["kind"] in ("energy", "screen"):
        lam = sec.hamiltonian(p["h"], p["eri"], p["e_nuc"], psi)
        E = float((psi.conj() * lam).real.sum()) / float((psi.conj() * psi).real.sum())
        if case["kind"] == "screen":
            return dict(energy=E, gradient=np.array([2.0 * sec.generator(op, lam, psi) for op in _pool(case)]))
        x = (sec.spread[1][:, None] | sec.spread[0]).reshape(-1).cpu().numpy()
        state = np.zeros(1 << case["n_qubits"], dtype="c16" if case["dtype"].startswith("c") else "f8")
        state[x] = psi.cpu().numpy()
        return dict(energy=E, state=state)
    E, g = _energy_gradient(sec, p, psi)
    if case["kind"] == "gradient":
        return dict(energy=E, gradient=g)
    amplitudes = psi[sec.index(_determinants(case))].cpu().numpy()
    if case["dtype"].startswith("c"):
        amplitudes = amplitudes.astype(np.complex128)
    return dict(energy=E, gradient=g, rdm=sec.rdm(psi), amplitudes=amplitudes)
