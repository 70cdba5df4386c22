"""Diagonal factors far from modulus 1 in register tiles: the compiler may keep
a factor aside only while its product with the others pending stays in a range
that FP32 tables and amplitudes hold.

CPU: exported programs with every table rounded to single precision, run by the
model of test_tile_program_cpu.py on a complex64 state.  GPU: the same circuits under the
plans that run tiles.  Tolerance, as in the tests of those plans: 1e-5 of the
largest amplitude (FP32 roundings, at most a few hundred per amplitude);
<sum Z> of a batch 1e-5 n of the norm.
"""
import math

import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C
from test_tile_program_cpu import CHUNK, CHUNK_UNITS, CSHEARS, END, GROUP, PH, RAMP, XCH, run_programs


def mat(q, m, **kw):
    return C.gate("u", q, mat=np.array(m, dtype=complex), **kw)


def non_unitary(family, n):
    layer = [C.gate("h", q) for q in range(n)]
    rng = np.random.default_rng(n)
    t, c = n - 1, n - 3
    if family == "growing":           # both entries, opposite directions
        return C.concat(layer + [mat(t, np.diag([math.exp(-0.5), math.exp(0.5)]))] * 100)
    if family == "half_x":            # tiny factor, then inverted by X
        return C.concat(layer + [mat(t, np.diag([1, 0.5]))] * 150 + [C.gate("x", t)] + layer)
    if family == "tenth_x":
        return C.concat(layer + [mat(3, np.diag([1, 0.1]))] * 40 + [C.gate("x", 3)] + layer)
    if family == "every_qubit":       # small common factor, large ones on the qubits
        return C.concat(layer + [mat(q, np.diag([0.01, 1])) for q in range(n)] * 2 + [C.gate("x", 2)])
    if family == "every_qubit_x":
        return C.concat(layer + [mat(q, np.diag([1, 1e-4])) for q in range(n)] + [C.gate("x", q) for q in range(n)])
    if family == "antidiagonal":
        return C.concat(layer + [mat(q, [[0, 1e-4], [1, 0]]) for q in range(n)] + [C.gate("t", 1)])
    if family == "pairs":             # controlled contractions, then X on both ends
        return C.concat(layer + [mat(t, np.diag([1, 0.5]), controls=(c,))] * 150 +
                        [mat(t, np.diag([0.5, 1]), controls=(2,))] * 100 + [C.gate("x", t), C.gate("x", c)])
    if family == "dense":             # not unitary, condition number 1e5, every qubit
        parts = list(layer)
        for q in range(n):
            a = C.haar_unitary_2x2(rng)
            parts += [mat(q, np.array([[1, 0.3], [0.2, 0.06001]])), mat(q, a @ np.diag([1, 0.4]) @ a.conj().T)]
        return C.concat(parts + [C.gate("x", q) for q in range(n)])
    if family == "scaled":            # multiples of unitary matrices that cancel out
        parts = list(layer)
        for q in range(n):
            parts.append(mat(q, 300.0 * C.haar_unitary_2x2(rng)))
        for q in range(n):
            parts.append(mat(q, C.haar_unitary_2x2(rng) / 300.0))
        return C.concat(parts)
    if family == "cooling":           # diagonals and rotations in turn
        parts = list(layer)
        for _ in range(12):
            for q in range(n):
                parts.append(mat(q, np.diag([math.exp(0.25), math.exp(-0.25)])))
                parts.append(C.gate("rz", q, params=(float(rng.uniform(0, 6)),)))
            parts += [C.gate("z", (q + 1) % n, controls=(q,)) for q in range(n)]
            parts.append(C.gate("ry", int(rng.integers(0, n)), params=(float(rng.uniform(0, 6)),)))
        return C.concat(parts)
    raise KeyError(family)


FAMILIES = ["growing", "half_x", "tenth_x", "every_qubit", "every_qubit_x", "antidiagonal", "pairs", "dense", "scaled",
            "cooling"]


def round_tables(words, info):
    """The programs' FP64 factors as FP32 has them (still stored as FP64)."""
    words = words.copy()
    for row in info:
        first, count, RB = int(row[0]), int(row[1]), int(row[3])
        units = words[first:first + count].reshape(-1, 4)
        RA, pc = 1 << RB, 0
        while True:
            f = int(units[pc][0])
            op, ln = f & 15, (f >> 4) & 0xFF
            if op == END:
                break
            if op == CHUNK:
                pc = (pc // CHUNK_UNITS + 1) * CHUNK_UNITS
                continue
            b = {GROUP: pc + 1 + (((f >> 24) & 31) + 1) // 2, RAMP: pc + 2, XCH: pc + 2, PH: pc + 3,
                 CSHEARS: pc + 1}.get(op, pc + ln)
            x = units[b:pc + ln].view(np.float64)
            with np.errstate(over="ignore"):
                x[...] = x.astype(np.float32)
            pc += ln
    return words


@pytest.mark.parametrize("n,tile", [(11, 11), (14, 11), (13, 12), (14, 13)])
@pytest.mark.parametrize("family", FAMILIES)
def test_programs_in_single_precision(orc, family, n, tile):
    from paper_1805_00988_gb300 import sim
    g = non_unitary(family, n)
    words, info = sim.sim_plan_tile_programs(n, 0, sim.to_sim_gates(g), tile)
    psi = C.random_state(n, seed=n + tile).astype(np.complex64)
    ref = orc.apply_circuit(psi.astype(np.complex128), g)
    assert np.max(np.abs(ref)) < 1e30
    with np.errstate(over="ignore", invalid="ignore"):
        got = run_programs(psi, n, round_tables(words, info), info)
    assert got.dtype == np.complex64
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))


# ------------------------------------------------------------------ GPU

@pytest.fixture(scope="module")
def gsim():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import sim as S
    return S


@pytest.mark.gpu
@pytest.mark.parametrize("plan,n,tile", [("staged", 11, 0), ("staged", 14, 12), ("staged", 14, 13), ("learned", 14, 0),
                                         ("learned", 19, 0)])
@pytest.mark.parametrize("family", FAMILIES)
def test_plans_match_oracle(gsim, orc, family, plan, n, tile):
    from paper_1805_00988_gb300 import costmodel
    g = non_unitary(family, n)
    psi = C.random_state(n, seed=n).astype(np.complex64)
    ref = orc.apply_circuit(psi.astype(np.complex128), g)
    st = gsim.State(n, "c64")
    model = costmodel.load()[0]
    gsim.sim_set_cost_model(st.h, model)
    st.load(psi)
    st.apply(g, plan=plan, **({"tile_qubits": tile} if tile else {}))
    got = st.state()
    st.close()
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [11, 12, 13])
def test_batch_matches_oracle(gsim, orc, tile):
    """<sum Z> (not divided by the norm) of each family, one tile and several passes."""
    circs = [(n, non_unitary(f, n)) for n in (9, 15) for f in FAMILIES]
    offs = np.concatenate([[0], np.cumsum([len(g) for _, g in circs])]).astype(np.int64)
    b = gsim.Batch([n for n, _ in circs], offs, C.concat([g for _, g in circs]), tile_qubits=tile)
    got = b.run()
    b.close()
    for (n, g), z in zip(circs, got):
        p = np.abs(orc.apply_circuit(orc.basis_state(n, 0), g)) ** 2
        w = n - 2 * np.array([bin(i).count("1") for i in range(1 << n)])
        assert abs(z - float(p @ w)) <= 1e-5 * n * p.sum()
