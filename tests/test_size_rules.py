"""The register sizes at which a call takes another kernel or plan, on both
sides of each line.

Tolerances: complex128 1e-11 of the largest amplitude and complex64 1e-5 (FP32
roundings of register tiles and per-gate kernels) or 1e-4 where fused blocks may
run, as in the tests of those plans; probabilities and collapsed states are compared
with one correctly rounded operation or two per value: 4 ulp.
"""
import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import sim as s
    return s


def mixed(n, seed):
    """Dense layers, swaps, diagonal stretches and controlled exchanges."""
    return C.concat([C.haar_cz(n, 2, seed=seed), C.random_gates(n, 3 * n, seed=seed), C.qft(n),
                     C.u3_cnot_ladder(n, 2, seed=seed), C.segments(n, ("rev", "phase", "graph"), 6 * n, seed=seed)])


@pytest.mark.parametrize("dt,n", [("c128", n) for n in (16, 17, 18, 20, 21)] + [("c64", n) for n in (16, 17, 18, 19)])
def test_per_gate_block_sizes(sim, orc, dt, n):
    """Small and large blocks; real, half-real and complex dense matrices, with and
    without controls."""
    g = C.concat([C.gate("h", 0), C.gate("h", n - 1), C.gate("ry", 3, params=(0.7,)), C.gate("rx", 2, params=(1.1,)),
                  C.gate("u3", n // 2, params=(0.3, 1.0, 2.0)), C.gate("h", 5, controls=(1,)),
                  C.gate("u3", 1, params=(2.0, 0.4, 0.9), controls=(n - 1, 4)), C.random_gates(n, 12, seed=n)])
    psi = C.random_state(n, seed=n)
    st = sim.State(n, dt)
    st.load(psi)
    st.apply(g, plan="per_gate")
    ref = orc.apply_circuit(psi.astype(st.np_dtype).astype(np.complex128), g)
    assert np.max(np.abs(st.state() - ref)) <= (1e-11 if dt == "c128" else 1e-5) * np.max(np.abs(ref))
    st.close()


@pytest.mark.parametrize("dt,plan,n", [("c64", "staged", n) for n in (18, 19)] + [("c64", "learned", n) for n in (12, 18, 19)] +
                         [("c128", "staged", n) for n in (19, 20)] + [("c128", "learned", n) for n in (11, 19, 20)])
def test_tile_sizes_match_oracle(sim, orc, dt, plan, n):
    from paper_1805_00988_gb300 import costmodel
    g = mixed(n, n)
    psi = C.random_state(n, seed=n + 1)
    st = sim.State(n, dt)
    model = costmodel.load()[0]
    sim.sim_set_cost_model(st.h, model)
    st.load(psi)
    st.apply(g, plan=plan)
    ref = orc.apply_circuit(psi.astype(st.np_dtype).astype(np.complex128), g)
    assert np.max(np.abs(st.state() - ref)) <= (1e-11 if dt == "c128" else 1e-5) * np.max(np.abs(ref))
    st.close()


@pytest.mark.parametrize("dt,n,k", [("c128", 21, 4), ("c128", 22, 4), ("c64", 26, 6)])
def test_mixed_plan_matches_per_gate(sim, dt, n, k):
    """Blocks and tiles in one call against complex128 gate by gate; the last gates are
    exchanges of places."""
    import torch
    from paper_1805_00988_gb300 import costmodel
    g = C.concat([mixed(n, 5), C.gate("swap", 0, target2=n - 1), C.gate("swap", 3, target2=9)])
    ref = sim.State(n, "c128")
    sim.sim_set_basis_state(ref.h, 5)
    ref.apply(g, plan="per_gate")
    st = sim.State(n, dt)
    model = costmodel.load()[0]
    sim.sim_set_cost_model(st.h, model)
    for plan, kw in (("fused", {"fuse_k": k}), ("learned", {})):
        sim.sim_set_basis_state(st.h, 5)
        st.apply(g, plan=plan, **kw)
        d = (st.tensor.to(torch.complex128) - ref.tensor).abs().max().item()
        assert d <= (1e-11 if dt == "c128" else 1e-4) * ref.tensor.abs().max().item(), plan
    st.close()
    ref.close()


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 11, 18])
def test_probabilities_and_collapse_vectors(sim, dt, n):
    """Output at an address that no 16-byte store may take; collapse on qubit 0 (inside
    a vector), 1 and the last."""
    import torch
    psi = C.random_state(n, seed=n).astype(np.complex64 if dt == "c64" else np.complex128)
    eps = np.finfo(psi.real.dtype).eps
    p64 = psi.real.astype(np.float64) ** 2 + psi.imag.astype(np.float64) ** 2
    st = sim.State(n, dt)
    st.load(psi)
    for real, tt in ((sim.SIM_F32, torch.float32), (sim.SIM_F64, torch.float64)):
        for shift in (0, 1, 3):
            buf = torch.full(((1 << n) + 8,), -1.0, dtype=tt, device="cuda")
            sim.sim_probabilities(st.h, buf[shift:].data_ptr(), real)
            torch.cuda.synchronize()
            got = buf.cpu().numpy().astype(np.float64)
            e = max(eps, np.finfo(np.float32).eps if real == sim.SIM_F32 else 0)
            assert np.all(np.abs(got[shift:shift + (1 << n)] - p64) <= 4 * e * p64 + 1e-45)
            assert np.all(got[:shift] == -1) and np.all(got[shift + (1 << n):] == -1)
    for q in sorted({0, min(1, n - 1), n - 1}):
        st.load(psi)
        m, pm = sim.sim_measure(st.h, q, 3)
        keep = ((np.arange(1 << n) >> q) & 1) == m
        want = np.where(keep, psi, 0) / np.sqrt(p64[keep].sum())
        got = st.state()
        assert abs(pm - p64[keep].sum()) <= 1e-6 and np.all(got[~keep] == 0)
        assert np.all(np.abs(got - want) <= 4 * eps * np.abs(want) + 1e-45)
    st.close()


def test_measured_halves_by_qubit(sim):
    """23 qubits: batches of 8 strided vectors, qubits inside a vector, below the
    stride, within the batch's span and above it.  Compensated sums: 1e-12 of the total."""
    n = 23
    psi = C.random_state(n, seed=n).astype(np.complex64)
    p = psi.real.astype(np.float64) ** 2 + psi.imag.astype(np.float64) ** 2
    st = sim.State(n, "c64")
    for q in (0, 1, 8, 9, 10, 11, 12, 13, n - 1):
        st.load(psi)
        m, pm = sim.sim_measure(st.h, q, 3)
        half = p.reshape(-1, 2, 1 << q)[:, m].sum()
        assert abs(pm - half / p.sum()) <= 1e-12
    st.close()
