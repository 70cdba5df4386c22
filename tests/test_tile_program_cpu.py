"""Tile programs (what the register-tile kernels run), checked without a GPU:
the words that sim_plan_tile_programs returns are run by a plain numpy model of
each operation, and the state must equal the FP64 oracle's for the original
circuit.  The model restates the operations from their description at the head
of csrc/tileprog.cuh: thread i and register k of a layout address one local
index; shears, tables, sign bits, ramps and masked operations act on physical
registers; the store sends exchanged labels to the other half of their pairs.

Tolerance: FP64 throughout, a few hundred gates of a few roundings each, on a
unit vector: 1e-12 per element."""
import math

import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C
from test_staged_encoding_cpu import phase_runs, reg_local

END, CHUNK, GROUP, RAMP, XCH, PH, CSHEARS, PERM = range(8)
CHUNK_UNITS = 512


THREADS = 128


def layout_index(M, RB, VEC, l):
    """local index of (thread, register): shape (128, 2^RB)"""
    regs = [reg_local(M, RB, VEC, l, j) for j in range(RB)]
    free = [b for b in range(M) if b not in regs]
    idx = np.zeros((THREADS, 1 << RB), dtype=np.int64)
    for i, b in enumerate(free):
        idx += ((np.arange(THREADS)[:, None] >> i) & 1) << b
    for j, b in enumerate(regs):
        idx += ((np.arange(1 << RB)[None, :] >> j) & 1) << b
    return idx


def run_tile(loc, units, RB, VEC, M, start, tile, tables):
    """One tile through a program; loc: the tile's amplitudes by local index.
    Returns (register array, layout)."""
    RA = 1 << RB
    tid = np.arange(THREADS)

    def lay(l):
        if l not in tables:
            tables[l] = layout_index(M, RB, VEC, l)
        return tables[l]

    layout = start
    v = loc[lay(layout)]
    zs = np.zeros(THREADS, dtype=np.int64)
    k = np.arange(RA)

    def shear(v, zs, j, a, bb):
        v = v.copy()
        s = (1 - 2 * ((zs >> j) & 1))[:, None]
        lo = k[((k >> j) & 1) == 0]
        v[:, lo] += s * a * v[:, lo | (1 << j)]
        v[:, lo | (1 << j)] += s * bb * v[:, lo]
        return v

    def cplx(u, cnt):
        return units[u:u + cnt].view(np.float64).reshape(-1, 2) @ np.array([1, 1j])

    pc = 0
    while True:
        h = units[pc]
        f = int(h[0])
        op, ln, arg = f & 15, (f >> 4) & 0xFF, f >> 12
        if op == END:
            break
        if op == CHUNK:
            pc = (pc // CHUNK_UNITS + 1) * CHUNK_UNITS
            continue
        assert pc // CHUNK_UNITS == (pc + ln) // CHUNK_UNITS, "an operation and the next header stay in one chunk"
        b = pc + 1
        tm, tv, om = int(h[1]) & 0xFF, (int(h[1]) >> 8) & 0xFF, int(h[2])
        ok = ((tid & tm) == tv) & ((tile & om) == om)
        if op in (RAMP, XCH, PH):
            km, kt = (int(x) for x in units[b].view(np.uint64))
            kbits = np.array([(km >> i) & 1 for i in range(RA)], dtype=bool)
            b += 1
        if op == GROUP:
            for e in range((f >> 24) & 31):
                w = units[b + e // 2][2 * (e % 2):2 * (e % 2) + 2]
                x, om = int(w[0]), int(w[1])
                on = ((tid & (x & 0xFF)) == ((x >> 8) & 0xFF)) & ((tile & om) == om)
                zs = np.where(on, zs ^ (x >> 16), zs)
            b += (((f >> 24) & 31) + 1) // 2
            kind, j = (f >> 12) & 7, (f >> 15) & 7
            hi = ((k >> j) & 1).astype(bool)[None, :]
            if kind == 1:
                v *= units[b:b + RA // 2].view(np.float64).ravel()[None, :]
                b += RA // 2
            elif kind == 2:
                v *= cplx(b, RA)[None, :]
                b += RA
            elif kind == 3:
                ta, tb = units[b:b + 1].view(np.float64).ravel()
                re, im = v.real + ta * v.imag, v.imag
                im = im + tb * re
                v = np.where(hi, (re + ta * im) + 1j * im, v)
                b += 1
            if (f >> 18) & 63:
                t = units[b:b + RB].view(np.float64).reshape(-1, 2)
                if not (f >> 29) & 1:
                    assert not zs.any()
                for j in range(RB):
                    if (f >> (18 + j)) & 1:
                        v = shear(v, zs, j, t[j, 0], t[j, 1])
            if (f >> 30) & 1:
                par = np.zeros((THREADS, RA), dtype=np.int64)
                for j in range(RB):
                    par ^= ((zs >> j) & 1)[:, None] & ((k >> j) & 1)[None, :]
                par ^= ((zs >> 6) & 1)[:, None]
                v = v * (1 - 2 * par)
                zs = np.zeros(THREADS, dtype=np.int64)
            lay_w = int(h[1])
            if f >> 31:
                assert not zs.any(), "signs are applied before the layout changes"
                assert layout == lay_w & 3
                loc = loc.copy()
                loc[lay(layout)] = v
                layout = lay_w >> 2
                v = loc[lay(layout)]
        elif op == PERM:
            assert not zs.any()
            assert layout == arg & 3
            loc = loc.copy()
            loc[lay(layout)] = v
            layout = arg >> 2
            slot = {(1 << x) + (((1 << x) >> (RB + 1)) << 1 if VEC == 2 else (1 << x) >> RB): x for x in range(M)}
            w = [slot[int(x)] for x in units[b:b + (7 + RB + 3) // 4].ravel()[:7 + RB]]
            src = np.zeros((THREADS, RA), dtype=np.int64)
            for i in range(7):
                src += (((tid >> i) & 1) << w[i])[:, None]
            for j in range(RB):
                src += (((k >> j) & 1) << w[7 + j])[None, :]
            v = loc[src]
        elif op == CSHEARS:
            c = cplx(b, 2)
            v = shear(v, zs, arg & 7, c[0], c[1])
        elif op == RAMP:
            f = np.ones(THREADS, dtype=np.complex128)
            g = np.ones(RA, dtype=np.complex128)
            u = b
            if arg & 8:
                g = cplx(u, RA)
                u += RA
            if arg & 16:
                t = cplx(u, 24)
                f = f * t[tid & 15] * t[16 + (tid >> 4)]
                u += 24
            for gi in range(6):
                if (arg >> (5 + gi)) & 1:
                    f = f * cplx(u, 16)[(tile >> (4 * gi)) & 15]
                    u += 16
            centre = arg & 7
            regs = ((k >> centre) & 1).astype(bool) if centre < 7 else kbits
            sel = ok[:, None] & regs[None, :]
            v = np.where(sel, v * f[:, None] * g[None, :], v)
        elif op == XCH:
            assert not zs.any()
            j, kind = arg & 7, (arg >> 3) & 3
            m = units[b:b + 4].view(np.float64).reshape(2, 2, 2) @ np.array([1, 1j])
            lo = k[(((k >> j) & 1) == 0) & kbits]
            x, y = v[:, lo].copy(), v[:, lo | (1 << j)].copy()
            if kind == 3:
                nx, ny = y, x
            else:
                nx, ny = m[0, 0] * x + m[0, 1] * y, m[1, 0] * x + m[1, 1] * y
            v[:, lo] = np.where(ok[:, None], nx, x)
            v[:, lo | (1 << j)] = np.where(ok[:, None], ny, y)
        elif op == PH:
            tt, ot, place = int(units[b][0]), int(units[b][1]), int(h[3])
            ad = cplx(b + 1, 2)
            if place:
                one = (((tid & (tt & 0xFF)) == (tt >> 8)) & ((tile & ot) == ot))[:, None] & np.ones(RA, dtype=bool)
            else:
                one = np.ones((THREADS, 1), dtype=bool) & np.array([(kt >> i) & 1 for i in range(RA)], dtype=bool)[None, :]
            cond = ok[:, None] & kbits[None, :]
            v = np.where(cond, v * np.where(one, ad[1], ad[0]), v)
        else:
            raise AssertionError("unknown operation %d" % op)
        pc += ln
    assert not zs.any(), "signs are applied before the store"
    return v, layout


def run_programs(psi, n, words, info):
    psi = psi.copy()
    for row in info:
        first, count, M, RB, VEC, start, end, flo, fhi, nh = (int(x) for x in row[:10])
        flip = (flo & 0xFFFFFFFF) | ((fhi & 0xFFFFFFFF) << 32)
        units = np.ascontiguousarray(words[first:first + count]).reshape(-1, 4)
        local = list(range(5)) + [int(q) for q in row[10:10 + nh]]
        outer = [q for q in range(n) if q not in local]
        lidx = np.arange(1 << M)
        gl = np.zeros(1 << M, dtype=np.int64)
        lflip = 0
        for b, q in enumerate(local):
            gl |= ((lidx >> b) & 1) << q
            lflip |= ((flip >> q) & 1) << b
        tables = {}
        for t in range(1 << (n - M)):
            base = sum(((t >> i) & 1) << q for i, q in enumerate(outer))
            v, layout = run_tile(psi[base | gl], units, RB, VEC, M, start, t, tables)
            assert layout == end
            if layout not in tables:
                tables[layout] = layout_index(M, RB, VEC, layout)
            out = np.empty(1 << M, dtype=np.complex128)
            out[tables[layout] ^ lflip] = v
            psi[base | gl] = out
    return psi


def single_precision(n, seed):
    """Unitaries whose entries were rounded to single precision, scaled and
    projector-like matrices, and real rotations."""
    rng = np.random.default_rng(seed)
    parts = []
    for _ in range(60):
        q = int(rng.integers(0, n))
        u = C.haar_unitary_2x2(rng)
        kind = int(rng.integers(0, 5))
        if kind == 0:
            u = u.astype(np.complex64).astype(np.complex128)
        elif kind == 1:
            u = 1.7 * u
        elif kind == 2:
            u = u @ np.diag([1.0, 0.6]) @ u.conj().T
        elif kind == 3:
            u = np.array([[1.0, 1.0], [1.0, 1.0]]) * 0.8
        ctrl = () if rng.random() < 0.7 else (int((q + 1 + rng.integers(0, n - 1)) % n),)
        parts.append(C.gate("u", q, controls=ctrl, mat=u))
        parts.append(C.gate("ry", int(rng.integers(0, n)), params=(float(rng.uniform(0, 7)),)))
    return C.concat(parts)


def clifford(n, seed):
    """H, X, Y, Z, S, CNOT, CZ, Toffoli and doubly controlled signs and phases:
    the label exchanges and the sign moves."""
    rng = np.random.default_rng(seed)
    parts = []
    for _ in range(220):
        qs = [int(x) for x in rng.permutation(n)[:3]]
        nm = ["h", "x", "y", "z", "s", "x", "z", "x", "z", "t", "y"][int(rng.integers(0, 11))]
        nc = int(rng.integers(0, 3)) if nm in ("x", "z", "t", "y") else 0
        parts.append(C.gate(nm, qs[0], controls=tuple(qs[1:1 + nc])))
    return C.concat(parts)


def circuit(family, n, seed):
    if family == "random":
        g = C.random_gates(n, 250, seed=seed, max_ctrl=2)
        sw = g["name"] == "swap"
        g["nctrl"][sw] = np.minimum(g["nctrl"][sw], 1)
        return g
    return {"haar": lambda: C.haar_cz(n, 5, seed=seed), "qft": lambda: C.concat([C.qft(n), C.qft_paper(n)]),
            "phase": lambda: C.phase_polynomial(n, 120, seed=seed), "ramps": lambda: phase_runs(n, seed),
            "ladder": lambda: C.u3_cnot_ladder(n, 4, seed=seed), "clifford": lambda: clifford(n, seed),
            "swaps": lambda: C.concat([C.reversible(n, 80, seed=seed), C.haar_cz(n, 1, seed=seed), C.phase_polynomial(n, 30, seed=seed),
                                       C.reversible(n, 60, seed=seed + 1)]),
            "variational": lambda: C.variational_layered(n, 4, np.random.default_rng(seed)),
            "matrices": lambda: single_precision(n, seed),
            "leftover": lambda: C.concat([C.gate("rz", n - 1, params=(0.3,)), C.gate("swap", 0, target2=n - 1)]),
            "hadamards": lambda: C.concat([C.gate("h", q) for q in list(range(n)) * 6])}[family]()


@pytest.mark.parametrize("family", ["random", "haar", "qft", "phase", "ramps", "ladder", "clifford", "variational", "swaps",
                                    "matrices", "hadamards", "leftover"])
@pytest.mark.parametrize("dtype,n,tile", [(0, 11, 11), (0, 14, 11), (0, 13, 12), (0, 14, 13), (1, 12, 11), (1, 14, 12)])
def test_programs_match_oracle(orc, family, dtype, n, tile):
    from paper_1805_00988_gb300 import sim
    gates = circuit(family, n, seed=n * 3 + tile + dtype)
    words, info = sim.sim_plan_tile_programs(n, dtype, sim.to_sim_gates(gates), tile)
    psi = C.random_state(n, seed=n + tile)
    ref = orc.apply_circuit(psi, gates)
    got = run_programs(psi, n, words, info)
    np.testing.assert_allclose(got, ref, atol=1e-12 * max(1.0, float(np.linalg.norm(ref))))


def test_permutations_need_no_arithmetic():
    """X, CNOT, Toffoli and SWAP compile to exchanges and label changes only,
    so they stay bit-exact."""
    from paper_1805_00988_gb300 import sim
    g = C.reversible(15, 200, seed=4)
    words, info = sim.sim_plan_tile_programs(15, 0, sim.to_sim_gates(g), 13)
    for row in info:
        units = words[row[0]:row[0] + row[1]].reshape(-1, 4)
        pc = 0
        while True:
            f = int(units[pc][0])
            op, ln = f & 15, (f >> 4) & 0xFF
            if op == END:
                break
            assert op in (XCH, CHUNK, PERM) or (op == GROUP and not (f >> 12) & 0x1FFFF)
            pc = (pc // CHUNK_UNITS + 1) * CHUNK_UNITS if op == CHUNK else pc + ln
