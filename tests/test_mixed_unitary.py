"""Only unitary circuits take the mixed form of the fused plan (blocks and register
tiles).  A plan described with multi-block passes asked for never mixes, so it gives the
blocks that a circuit with a contraction must run as, and on the GPU the same bits."""
import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C


def mat(q, m, **kw):
    return C.gate("u", q, mat=np.array(m, dtype=complex), **kw)


def extra(kind, n):
    rng = np.random.default_rng(5)
    a, b = C.haar_unitary_2x2(rng), C.haar_unitary_2x2(rng)
    return {"none": [], "single_precision": [mat(3, a.astype(np.complex64))],
            "contraction": [mat(3, np.diag([1, 0.5]))],
            "projector": [mat(n - 1, np.diag([1, 0]))],
            "dense_contraction": [mat(4, a @ np.diag([1, 0.3]) @ b)],
            "controlled_contraction": [mat(2, np.diag([0.2, 1]), controls=(6,))],
            "shear": [mat(2, [[1, 0.1], [0, 1]])],
            "grown": [mat(2, np.diag([1, 2.0]))]}[kind]


def circuit(kind, n):
    return C.concat([C.qft(n), *extra(kind, n), C.qft(n), C.phase_polynomial(n, 40, seed=2)])


@pytest.mark.parametrize("dtype,n,k", [(0, 26, 6), (1, 22, 4)])
@pytest.mark.parametrize("kind", ["none", "single_precision", "contraction", "projector", "dense_contraction",
                                  "controlled_contraction", "shear", "grown"])
def test_only_unitary_circuits_mix(kind, dtype, n, k):
    from paper_1805_00988_gb300 import sim
    g = sim.to_sim_gates(circuit(kind, n))
    got = sim.sim_plan_describe(n, dtype, g, sim.plan_opts("fused", fuse_k=k))[:2]
    blocks = sim.sim_plan_describe(n, dtype, g, sim.plan_opts("fused", fuse_k=k, flags=sim.SIM_FLAG_MULTI_BLOCK_PASSES))[:2]
    assert blocks[0] == blocks[1] > 0
    if kind in ("none", "single_precision"):
        assert got[1] < blocks[1]              # tiles took the QFTs
    else:
        assert got == blocks


@pytest.mark.gpu
@pytest.mark.parametrize("dt,n,k", [("c64", 26, 6), ("c128", 22, 4), ("c128", 14, 4)])
@pytest.mark.parametrize("kind", ["contraction", "projector", "controlled_contraction"])
def test_contractions_run_in_blocks(dt, n, k, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import costmodel, sim
    g = C.concat([circuit(kind, n), *extra("contraction", n) * 60, C.gate("x", 3)])
    st = sim.State(n, dt)
    model = costmodel.load()[0]
    sim.sim_set_cost_model(st.h, model)
    sim.sim_set_basis_state(st.h, 5)
    st.apply(g, plan="fused", fuse_k=k, flags=sim.SIM_FLAG_MULTI_BLOCK_PASSES)
    blocks = st.tensor.clone()
    sim.sim_profile_enable(st.h, True)
    for plan, kw in (("fused", {"fuse_k": k}), ("learned", {})):
        sim.sim_set_basis_state(st.h, 5)
        st.apply(g, plan=plan, **kw)
        assert "staged" not in sim.sim_profile_read(st.h)
        assert torch.equal(st.tensor, blocks), plan
    st.close()
