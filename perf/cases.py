"""What this library is asked to do, as timed cases.

Each case is one call a user's program makes through the public entry points
(paper_1805_00988_gb300.sim): a circuit applied to a register from a basis
state under one of the plans, a noisy circuit on a density matrix, a batch of
small parameterised circuits, or the read-out of a finished state.  Sizes are
those of the repository's own workloads (QFT-28, Haar/CZ layers at 30 qubits,
the 14-qubit U3 + CNOT ladder, variational circuits of 8..20 qubits, noisy
density matrices) and of its mid-size test circuits.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the register, circuit and buffers a program holds
    run(state)          one call (or the few that belong together)
    work(case)          bytes and flops the result cannot do without
    exact(case, seed)   the same result in 64 bits, from torch alone
"""
import functools
import math

import numpy as np
import torch

from paper_1805_00988_gb300 import circuits as C
from paper_1805_00988_gb300 import costmodel, sim

MIXES = {"mix_haar_graph": ("haar", "graph", "haar", "graph"), "mix_graph_qft_haar": ("graph", "qft", "haar"),
         "mix_rev_phase_ladder": ("rev", "phase", "ladder", "graph")}


def listed():
    return [
        # the smallest call: the 14-qubit worked example, 30-odd launches on a
        # 128 KiB state (launch latency), with its probabilities
        {"name": "bv_14q_c64_per_gate", "kind": "circuit", "family": "bv", "n": 14, "depth": 1, "dtype": "c64",
         "plan": "per_gate", "k": 0, "probs": True},
        # the plain method's own configuration: 14 qubits, complex128, 20
        # layers of U3 and CNOT ladders, state and probabilities
        {"name": "ladder_14q_c128_per_gate", "kind": "circuit", "family": "ladder", "n": 14, "depth": 20,
         "dtype": "c128", "plan": "per_gate", "k": 0, "probs": True},
        # the paper's benchmark circuit at its largest size, one kernel a gate
        {"name": "qft_28q_c64_per_gate", "kind": "circuit", "family": "qft", "n": 28, "depth": 1, "dtype": "c64",
         "plan": "per_gate", "k": 0, "probs": False},
        # the same circuit as a user who wants it fast runs it, both precisions
        {"name": "qft_28q_c64_learned", "kind": "circuit", "family": "qft", "n": 28, "depth": 1, "dtype": "c64",
         "plan": "learned", "k": 0, "probs": False},
        {"name": "qft_27q_c128_learned", "kind": "circuit", "family": "qft", "n": 27, "depth": 1, "dtype": "c128",
         "plan": "learned", "k": 0, "probs": False},
        # the headline workload: 30 qubits, depth 20, the learned plan, with
        # the norm its user checks afterwards
        {"name": "haar_30q_c64_learned", "kind": "circuit", "family": "haar", "n": 30, "depth": 20, "dtype": "c64",
         "plan": "learned", "k": 0, "probs": False},
        # a mid-size register, where most interactive work happens
        {"name": "haar_20q_c64_learned", "kind": "circuit", "family": "haar", "n": 20, "depth": 20, "dtype": "c64",
         "plan": "learned", "k": 0, "probs": True},
        # stretches of different gate families, an odd size, register tiles
        {"name": "mix_23q_c64_staged", "kind": "circuit", "family": "mix_rev_phase_ladder", "n": 23, "depth": 10,
         "dtype": "c64", "plan": "staged", "k": 0, "probs": False},
        # double precision at a size that fills the chip (tensor-core digits)
        {"name": "haar_26q_c128_learned", "kind": "circuit", "family": "haar", "n": 26, "depth": 20, "dtype": "c128",
         "plan": "learned", "k": 0, "probs": False},
        # many small parameterised circuits, one value each (a variational
        # optimiser's inner loop)
        {"name": "batch_1024_8to20q", "kind": "batch", "count": 1024, "nmin": 8, "nmax": 20, "lmin": 4, "lmax": 12},
        # noisy circuit on a density matrix: gates and channels
        {"name": "density_13q_c64_learned", "kind": "density", "n": 13, "depth": 10, "dtype": "c64",
         "plan": "learned"},
        # a finished state read out: probabilities, a million shots with norm
        # and <sum Z>, then one qubit measured
        {"name": "readout_28q_c64", "kind": "readout", "n": 28, "dtype": "c64", "shots": 1000000},
    ]


def draw(rng):
    """One more case: kinds, sizes, dtypes and plans spread over the range of
    the listed ones (register sizes are drawn as qubit counts, the logarithm
    of the state)."""
    r = rng.random()
    if r < 0.62:
        dtype = "c64" if rng.random() < 0.7 else "c128"
        plan = rng.choice(["learned", "learned", "learned", "per_gate", "staged", "fused"])
        top = {"per_gate": 25, "staged": 27, "fused": 28, "learned": 28}[plan] if dtype == "c64" else \
              {"per_gate": 22, "staged": 22, "fused": 25, "learned": 25}[plan]
        n = rng.randint(14 if plan == "fused" else 10, top)
        k = 0
        if plan == "fused":
            k = rng.choice([4, 5, 6]) if dtype == "c64" else 4
        fam = rng.choice(["haar", "qft", "qft_paper", "ladder", "variational"] + sorted(MIXES))
        return {"kind": "circuit", "family": fam, "n": n, "depth": rng.randint(3, 20), "dtype": dtype, "plan": plan,
                "k": k, "probs": n <= 20 and rng.random() < 0.5}
    if r < 0.78:
        nmin = rng.randint(4, 12)
        lmin = rng.randint(1, 6)
        return {"kind": "batch", "count": int(round(math.exp(rng.uniform(math.log(64), math.log(1024))))),
                "nmin": nmin, "nmax": rng.randint(nmin, 20), "lmin": lmin, "lmax": rng.randint(lmin, 12)}
    if r < 0.88:
        return {"kind": "density", "n": rng.randint(7, 13), "depth": rng.randint(2, 10), "dtype": "c64",
                "plan": rng.choice(["learned", "fused"])}
    return {"kind": "readout", "n": rng.randint(14, 28), "dtype": rng.choice(["c64", "c64", "c128"]),
            "shots": int(round(math.exp(rng.uniform(math.log(1000), math.log(1000000)))))}


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=1)
def _model():
    """The shipped plan cost model, loaded once per program."""
    return costmodel.load()[0]


def _gates(case, seed):
    n, d, fam = case["n"], case["depth"], case["family"]
    if fam == "bv":
        return C.bernstein_vazirani(n, C.random_basis_index(n, seed))
    if fam == "haar":
        return C.haar_cz(n, d, seed=seed)
    if fam == "ladder":
        return C.u3_cnot_ladder(n, d, seed=seed)
    if fam == "qft":
        return C.qft(n)
    if fam == "qft_paper":
        return C.qft_paper(n)
    if fam == "variational":
        return C.variational_layered(n, d, np.random.default_rng(seed))
    return C.segments(n, MIXES[fam], max(2 * n, d * n // 2), seed=seed)


def _start(case, seed):
    """The basis state a circuit starts from: the QFT transforms a seeded
    index (the paper's benchmark), the others start in |0...0>."""
    return C.random_basis_index(case["n"], seed) if case["family"] in ("qft", "qft_paper") else 0


def _random_state(n, dtype, seed):
    """Complex normal amplitudes, normalised: what a deep random circuit leaves."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    rd = torch.float32 if dtype == "c64" else torch.float64
    v = torch.empty((1 << n, 2), dtype=rd, device="cuda").normal_(generator=g).mul_(math.sqrt(0.5 / (1 << n)))
    return torch.view_as_complex(v)


def prepare(case, seed):
    s = {"case": case}
    kind = case["kind"]
    if kind == "batch":
        ns, offs, g = C.variational(case["count"], case["nmin"], case["nmax"], case["lmin"], case["lmax"], seed=seed)
        s["batch"] = sim.Batch(ns, offs, sim.to_sim_gates(g))
    elif kind == "density":
        s["rho"] = sim.DensityMatrix(case["n"], case["dtype"])
        s["gates"] = sim.to_sim_gates(C.noisy_haar_cz(case["n"], case["depth"], seed=seed))
        if case["plan"] == "learned":
            sim.sim_set_cost_model(s["rho"].h, _model())
        s["opts"] = sim.plan_opts(case["plan"])
    elif kind == "readout":
        s["reg"] = sim.State(case["n"], case["dtype"])
        s["psi"] = _random_state(case["n"], case["dtype"], seed)
        s["probs"] = torch.empty(1 << case["n"], dtype=torch.float32 if case["dtype"] == "c64" else torch.float64,
                                 device="cuda")
        s["shots"] = torch.empty(case["shots"], dtype=torch.int64, device="cuda")
        s["seed"], s["qubit"] = int(seed), int(seed) % case["n"]
    else:
        s["reg"] = sim.State(case["n"], case["dtype"])
        s["gates"] = sim.to_sim_gates(_gates(case, seed))
        s["start"] = _start(case, seed)
        if case["plan"] == "learned":
            sim.sim_set_cost_model(s["reg"].h, _model())
        s["opts"] = sim.plan_opts(case["plan"], fuse_k=case["k"])
        if case["probs"]:
            s["probs"] = torch.empty(1 << case["n"], dtype=torch.float32 if case["dtype"] == "c64" else torch.float64,
                                     device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        # complex64 registers: the values carry single precision and go into
        # a single-precision optimiser
        return {"expz": s["batch"].run().astype(np.float32)}
    if kind == "density":
        rho = s["rho"]
        rho.set_basis(0)
        sim.sim_dm_apply_circuit(rho.h, s["gates"], s["opts"])
        return {"rho": rho.tensor, "trace": rho.trace()}
    real = sim.SIM_F32 if case["dtype"] == "c64" else sim.SIM_F64
    reg = s["reg"]
    if kind == "readout":
        sim.sim_load_state(reg.h, s["psi"].data_ptr(), False)
        sim.sim_probabilities(reg.h, s["probs"].data_ptr(), real)
        _, norm, expz = sim.sim_sample_observe(reg.h, case["shots"], s["seed"], out=s["shots"].data_ptr(),
                                               out_on_device=True)
        outcome, prob = sim.sim_measure(reg.h, s["qubit"], s["seed"])
        return {"probs": s["probs"], "shots": s["shots"], "observed": np.array([norm, expz, prob]),
                "outcome": outcome, "state": reg.tensor}
    sim.sim_set_basis_state(reg.h, s["start"])
    sim.sim_apply_circuit(reg.h, s["gates"], s["opts"])
    out = {"state": reg.tensor}
    if case["probs"]:
        sim.sim_probabilities(reg.h, s["probs"].data_ptr(), real)
        out["probs"] = s["probs"]
    if case["n"] >= 30:
        out["norm"] = sim.sim_norm(reg.h)
    return out


# ---------------------------------------------------------------- work
#: real flops per amplitude of one uncontrolled gate: a full 2 x 2 is two
#: complex multiply-adds, a real one half of that, RZ one complex multiply, a
#: phase on |1> half of that, a sign or a move nothing
_FLOPS = {"u": 16, "u3": 16, "rx": 16, "ry": 8, "h": 8, "y": 0, "rz": 6, "p": 3, "t": 3, "tdg": 3, "s": 0, "sdg": 0,
          "x": 0, "z": 0, "swap": 0, "dep": 8, "adamp": 8}


def _flops(g, n):
    f = np.zeros(len(g))
    for nm, v in _FLOPS.items():
        f[g["name"] == nm] = v
    return float(np.sum(f * np.exp2(n - g["nctrl"].astype(float))))


def work(case):
    amp = 16 if case.get("dtype") == "c128" else 8
    if case["kind"] == "batch":
        ns, offs, g = C.variational(case["count"], case["nmin"], case["nmax"], case["lmin"], case["lmax"], seed=1)
        fl = sum(_flops(g[offs[i]:offs[i + 1]], int(ns[i])) for i in range(len(ns)))
        # in: one angle per rotation; out: one value per circuit
        return {"bytes": 8.0 * float(np.sum(g["name"] != "z")) + 8.0 * case["count"], "flops": fl}
    n = case["n"]
    if case["kind"] == "density":
        g = C.noisy_haar_cz(n, case["depth"], seed=1)
        gate = np.isin(g["name"], ("dep", "adamp"), invert=True)
        return {"bytes": float(amp) * 4.0 ** n, "flops": 2 * _flops(g[gate], 2 * n) + _flops(g[~gate], 2 * n)}
    state = float(amp) * 2.0 ** n
    if case["kind"] == "readout":
        # in: the state; out: probabilities, shots and the collapsed state
        return {"bytes": 2 * state + state / 2 + 8.0 * case["shots"], "flops": 3.0 * 2.0 ** n}
    g = _gates(case, 1)
    return {"bytes": state + (state / 2 if case["probs"] else 0.0), "flops": _flops(g, n)}


# ---------------------------------------------------------------- 64-bit reference
_R2 = math.sqrt(0.5)


def _matrix(name, p, mat):
    th, ph, la = (float(x) for x in p)
    c, s = math.cos(th / 2), math.sin(th / 2)
    e = lambda a: complex(math.cos(a), math.sin(a))  # noqa: E731
    if name == "u":
        return [complex(mat[2 * i], mat[2 * i + 1]) for i in range(4)]
    return {"x": [0, 1, 1, 0], "y": [0, -1j, 1j, 0], "z": [1, 0, 0, -1], "h": [_R2, _R2, _R2, -_R2],
            "s": [1, 0, 0, 1j], "sdg": [1, 0, 0, -1j], "t": [1, 0, 0, complex(_R2, _R2)],
            "tdg": [1, 0, 0, complex(_R2, -_R2)], "rx": [c, -1j * s, -1j * s, c], "ry": [c, -s, s, c],
            "rz": [e(-th / 2), 0, 0, e(th / 2)], "p": [1, 0, 0, e(th)],
            "u3": [c, -e(la) * s, e(ph) * s, e(ph + la) * c]}[name]


def _halves(psi, n, t, controls):
    """Views of the amplitudes with qubit t at 0 and at 1, controls at 1."""
    qs = sorted((t,) + tuple(controls), reverse=True)
    shape, index, above = [], [], n
    for q in qs:
        shape += [1 << (above - 1 - q), 2]
        index += [slice(None), None if q == t else 1]
        above = q
    shape.append(1 << above)
    index.append(slice(None))
    v = psi.view(shape)
    return v[tuple(0 if i is None else i for i in index)], v[tuple(1 if i is None else i for i in index)]


def _apply2(psi, n, t, controls, m):
    lo, hi = _halves(psi, n, t, controls)
    a, b, c, d = (complex(x) for x in m)
    if b == 0 and c == 0:
        if a != 1:
            lo.mul_(a)
        if d != 1:
            hi.mul_(d)
        return
    new = a * lo + b * hi
    hi.mul_(d).add_(lo * c)
    lo.copy_(new)


def _apply_all(psi, n, gates):
    for g in gates:
        name, t = str(g["name"]), int(g["target"])
        cs = tuple(int(c) for c in g["ctrl"][:int(g["nctrl"])])
        if name == "swap":
            o = int(g["target2"])
            for a, b, more in ((o, t, ()), (t, o, cs), (o, t, ())):   # three CNOTs: control a, target b
                _apply2(psi, n, b, (a,) + more, [0, 1, 1, 0])
        else:
            _apply2(psi, n, t, cs, _matrix(name, g["params"], g["mat"]))


def _basis(n, j):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[j] = 1
    return psi


def _exact_qft(n, j):
    """sum_k e^{2 pi i j k / 2^n} |k> / sqrt(2^n)."""
    N = 1 << n
    out = torch.empty(N, dtype=torch.complex128, device="cuda")
    for o in range(0, N, 1 << 24):
        k = torch.arange(o, min(N, o + (1 << 24)), dtype=torch.int64, device="cuda")
        th = (k * j % N).to(torch.float64) * (2 * math.pi / N)
        out[o:o + len(k)] = torch.polar(torch.full_like(th, 1 / math.sqrt(N)), th)
    return out


def _exact_batch(case, seed):
    """All circuits of one register size at once: a (circuits, 2^n) array,
    rotations with a matrix per circuit, finished circuits left alone."""
    ns, offs, g = C.variational(case["count"], case["nmin"], case["nmax"], case["lmin"], case["lmax"], seed=seed)
    out = np.zeros(len(ns))
    for n in sorted(set(int(v) for v in ns)):
        ids_all = np.nonzero(ns == n)[0]
        ring = n if n > 2 else n - 1
        x = torch.arange(1 << n, device="cuda")
        pop = sum((x >> q) & 1 for q in range(n))
        flips = sum(((x >> q) & 1) * ((x >> ((q + 1) % n)) & 1) for q in range(ring))
        cz = (1 - 2 * (flips % 2)).to(torch.float64)
        per = max(1, (1 << 27) >> n)
        for i0 in range(0, len(ids_all), per):
            ids = ids_all[i0:i0 + per]
            layers = np.array([(offs[i + 1] - offs[i]) // (2 * n + ring) for i in ids])
            psi = torch.zeros((len(ids), 1 << n), dtype=torch.complex128, device="cuda")
            psi[:, 0] = 1
            for layer in range(int(layers.max())):
                live = np.nonzero(layers > layer)[0]
                th = np.zeros((len(ids), n, 2))
                for i in live:
                    f = offs[ids[i]] + layer * (2 * n + ring)
                    th[i] = g["params"][f:f + 2 * n, 0].reshape(n, 2)
                th = torch.from_numpy(th).cuda()
                for q in range(n):
                    v = psi.view(len(ids), -1, 2, 1 << q)
                    c, s = torch.cos(th[:, q, 0] / 2)[:, None, None], torch.sin(th[:, q, 0] / 2)[:, None, None]
                    e = torch.polar(torch.ones_like(c), th[:, q, 1][:, None, None] / 2)
                    lo, hi = v[:, :, 0], v[:, :, 1]
                    new = (c * lo - s * hi) * e.conj()
                    hi.copy_((s * lo + c * hi) * e)
                    lo.copy_(new)
                live_t = torch.from_numpy((layers > layer).astype(np.float64)).cuda()[:, None]
                psi *= cz[None, :] * live_t + (1 - live_t)
            out[ids] = ((psi.real ** 2 + psi.imag ** 2) @ (n - 2 * pop).to(torch.float64)).cpu().numpy()
    return out


def _superop(name, p):
    """The channel on (row bit, column bit) as a 4 x 4 matrix over index
    2 * row + column."""
    if name == "dep":
        ks = [math.sqrt(1 - 0.75 * p) * np.eye(2), math.sqrt(p / 4) * np.array([[0, 1], [1, 0]]),
              math.sqrt(p / 4) * np.array([[0, -1j], [1j, 0]]), math.sqrt(p / 4) * np.diag([1, -1])]
    else:
        ks = [np.diag([1, math.sqrt(1 - p)]), np.array([[0, math.sqrt(p)], [0, 0]])]
    return sum(np.kron(k, np.conj(k)) for k in ks)


def _exact_density(case, seed):
    n, N = case["n"], 2 * case["n"]
    rho = _basis(N, 0)
    for g in C.noisy_haar_cz(n, case["depth"], seed=seed):
        name, t = str(g["name"]), int(g["target"])
        if name in ("dep", "adamp"):
            S = torch.from_numpy(np.asarray(_superop(name, float(g["params"][0])), dtype=np.complex128)).cuda()
            v = rho.view(1 << (n - 1 - t), 2, 1 << (n - 1), 2, 1 << t)
            x = [v[:, r, :, c] for r in (0, 1) for c in (0, 1)]
            y = [sum(S[i, j] * x[j] for j in range(4) if S[i, j] != 0) for i in range(4)]
            for i in range(4):
                x[i].copy_(y[i])
            continue
        cs = tuple(int(c) for c in g["ctrl"][:int(g["nctrl"])])
        m = _matrix(name, g["params"], g["mat"])
        _apply2(rho, N, t + n, tuple(c + n for c in cs), m)
        _apply2(rho, N, t, cs, [complex(z).conjugate() for z in m])
    diag = rho.view(1 << n, 1 << n).diagonal().real
    return {"rho": rho, "trace": float(diag.sum())}


def _exact_readout(case, seed):
    n = case["n"]
    psi = _random_state(n, case["dtype"], seed).to(torch.complex128)
    p = psi.real ** 2 + psi.imag ** 2
    norm = float(p.sum())
    x = torch.arange(1 << n, device="cuda")
    w = torch.full((1 << n,), float(n), dtype=torch.float64, device="cuda")
    for q in range(n):
        w -= 2.0 * ((x >> q) & 1)
    expz = float((p * w).sum())
    del w, x
    q = int(seed) % n
    halves = psi.view(-1, 2, 1 << q)
    ph = [float((halves[:, b].real ** 2 + halves[:, b].imag ** 2).sum()) for b in (0, 1)]
    # the measurement draw: SplitMix64 of the seed (Steele, Lea and Flood 2014)
    mask = (1 << 64) - 1
    z = (int(seed) + 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    u = ((z ^ (z >> 31)) >> 11) * 2.0 ** -53
    outcome = 0 if ph[0] > u * (ph[0] + ph[1]) else 1
    halves[:, 1 - outcome] = 0
    halves[:, outcome] *= 1 / math.sqrt(ph[outcome])
    return {"probs": p, "shots": None, "observed": np.array([norm, expz, ph[outcome] / (ph[0] + ph[1])]),
            "outcome": None, "state": psi}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return {"expz": _exact_batch(case, seed)}
    if kind == "density":
        return _exact_density(case, seed)
    if kind == "readout":
        return _exact_readout(case, seed)
    n = case["n"]
    if n > 28 or (n > 26 and case["family"] != "qft"):
        return None      # a minute and more in 64 bits
    if case["family"] == "qft":
        psi = _exact_qft(n, _start(case, seed))
    else:
        psi = _basis(n, _start(case, seed))
        _apply_all(psi, n, _gates(case, seed))
    out = {"state": psi}
    if case["probs"]:
        out["probs"] = psi.real ** 2 + psi.imag ** 2
    return out
