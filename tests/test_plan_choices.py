"""Circuits that the large-register plans must run in blocks, and in tiles: choices that
measured slower the other way (the figures stand at the rules).

GPU tolerances: those of the plans' tests, 1e-11 (complex128) and 1e-4 (complex64 blocks)
of the largest amplitude."""
import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C


def controlled_u3(n, m, seed):
    rng = np.random.default_rng(seed)
    parts = []
    for _ in range(m):
        a, b = (int(x) for x in rng.permutation(n)[:2])
        parts.append(C.gate("u3", a, controls=(b,) if rng.random() < 0.7 else (), params=tuple(rng.uniform(0, 6, 3))))
    return C.concat(parts)


@pytest.mark.parametrize("dtype,n,k,kind,blocks", [
    (1, 24, 4, "phases", True), (1, 27, 4, "phases", True), (1, 27, 4, "qft", False), (1, 22, 4, "ladder", True),
    (1, 22, 4, "reversible", False), (0, 26, 6, "ladder", True), (0, 26, 6, "controlled_u3", True),
    (0, 26, 6, "reversible", False), (0, 27, 6, "phases", False), (0, 28, 6, "one", False), (0, 28, 6, "haar", True)])
def test_fused_plan_runs_blocks_or_tiles(dtype, n, k, kind, blocks):
    from paper_1805_00988_gb300 import sim
    g = {"phases": lambda: C.phase_polynomial(n, 80, seed=1), "qft": lambda: C.qft(n, swaps=False),
         "ladder": lambda: C.u3_cnot_ladder(n, 3, seed=1), "reversible": lambda: C.reversible(n, 60, seed=1),
         "controlled_u3": lambda: controlled_u3(n, 60, 1), "one": lambda: C.gate("h", 0),
         "haar": lambda: C.haar_cz(n, 6, seed=1)}[kind]()
    passes, nb = sim.sim_plan_describe(n, dtype, sim.to_sim_gates(g), sim.plan_opts("fused", fuse_k=k))[:2]
    assert (nb == passes) if blocks else (nb == 0 and passes > 0)


@pytest.mark.gpu
@pytest.mark.parametrize("dt,n,kind,staged", [("c128", 14, "controlled_u3", False), ("c128", 14, "ladder", True),
                                              ("c64", 25, "ladder", False), ("c64", 25, "controlled_u3", False),
                                              ("c64", 25, "haar", True), ("c64", 24, "ladder", True)])
def test_learned_plan_runs_blocks_or_tiles(dt, n, kind, staged):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import costmodel, sim
    g = {"ladder": lambda: C.u3_cnot_ladder(n, 3, seed=1), "controlled_u3": lambda: controlled_u3(n, 60, 1),
         "haar": lambda: C.haar_cz(n, 4, seed=1)}[kind]()
    g = C.concat([g, C.gate("swap", 0, target2=n - 1)])
    ref = sim.State(n, "c128")
    ref.apply(g, plan="per_gate")
    st = sim.State(n, dt)
    model = costmodel.load()[0]
    sim.sim_set_cost_model(st.h, model)
    sim.sim_profile_enable(st.h, True)
    st.apply(g, plan="learned")
    prof = sim.sim_profile_read(st.h)
    if staged:
        assert not any(k.startswith("fused") for k in prof)
    else:
        assert any(k.startswith("fused") for k in prof)
        if dt == "c64":
            assert "staged" not in prof and set(sim.sim_last_plan(st.h)) == {6}
    d = (st.tensor.to(torch.complex128) - ref.tensor).abs().max().item()
    assert d <= (1e-11 if dt == "c128" else 1e-4) * ref.tensor.abs().max().item()
    st.close()
    ref.close()
