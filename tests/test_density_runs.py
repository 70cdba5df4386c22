"""Channels between gates under the staged plan: one matrix per qubit, two
qubits a pass (k_channels), gates on other qubits moved before them.  Against
the FP64 density oracle and against the per-gate plan, which applies every
record in order, one channel a pass.

Tolerances, element-wise relative to max |rho|: complex128 1e-11; complex64
1e-5 (as in test_density.py: at most 90 records of a few FP32 roundings,
6e-8 each).  Trace: every channel preserves it, and a channel's 1 - p is applied as
a difference, so only unbiased roundings of the sums are left: 1e-6 after 96
channels (rounded coefficients would lose 3e-8 with each, 2.9e-6).
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


def runs(n, seed):
    """Layers of gates on some qubits and channels on others, several on one
    qubit, with p = 0, p = 1 and the middle of the range."""
    rng = np.random.default_rng(seed)
    parts = []
    for layer in range(4):
        parts.append(C.random_gates(n, 4, seed=seed + layer))
        for _ in range(2 * n + 1):
            p = float(rng.choice([0.0, 1e-3, 0.3, 0.9, 1.0], p=[0.1, 0.4, 0.3, 0.1, 0.1]))
            parts.append(C.channel(str(rng.choice(C.CHANNEL_NAMES)), int(rng.integers(0, n)), p))
            if rng.random() < 0.3:
                parts.append(C.random_gates(n, 1, seed=int(rng.integers(1 << 30))))
    return C.concat(parts)


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 6, 7])
def test_channel_runs_match_oracle(sim, orc, dt, n):
    from oracle import density as dm
    g = runs(n, 17 * n)
    rng = np.random.default_rng(n)
    G = rng.standard_normal((1 << n, 3)) + 1j * rng.standard_normal((1 << n, 3))
    rho = G @ G.conj().T
    rho /= np.trace(rho).real
    ref = dm.apply_circuit(rho.astype(np.complex64).astype(np.complex128) if dt == "c64" else rho, g)
    for plan in ("staged", "per_gate"):
        st = sim.DensityMatrix(n, dt)
        st.load(rho)
        st.apply(g, plan=plan)
        err = np.max(np.abs(st.matrix().astype(np.complex128) - ref))
        assert err <= (1e-11 if dt == "c128" else 1e-5) * np.max(np.abs(ref)), (plan, err)
        st.close()


def test_trace_is_kept(sim):
    n = 8
    st = sim.DensityMatrix(n, "c64")
    g = C.noisy(C.concat([C.gate("h", q) for q in range(n)]), n, n, channels=(("dep", 1e-3), ("adamp", 2e-3)) * 6)
    for plan in ("staged", "per_gate"):
        st.set_basis(0)
        st.apply(g, plan=plan)
        assert abs(st.trace() - 1.0) < 1e-6, plan
    st.close()
