"""What the introspection calls say about a plan is what a run does: the tile size
that is taken when the caller leaves it open, the tile passes, and the passes of a
fused plan that mixes blocks and tiles.  All comparisons are of whole numbers."""
import numpy as np
import pytest

from paper_1805_00988_gb300 import circuits as C


def default_tile(n, c128):
    if c128:
        return 12 if n >= 20 else 11
    return 11 if n <= 18 else 12 if n <= 22 else 13


def sample(n, seed):
    """Swaps (renamed in a run), diagonal stretches, rotations and exchanges."""
    return C.concat([C.haar_cz(n, 2, seed=seed), C.gate("swap", 0, target2=n - 1), C.phase_polynomial(n, 2 * n, seed=seed),
                     C.reversible(n, 3 * n, seed=seed), C.qft(n)])


@pytest.mark.parametrize("c128", [0, 1])
@pytest.mark.parametrize("n", [11, 12, 14, 18, 19, 20, 22, 23])
def test_open_tile_size_is_the_one_that_runs(n, c128):
    from paper_1805_00988_gb300 import sim
    g, t = sim.to_sim_gates(sample(n, n)), default_tile(n, c128)
    words, info = sim.sim_plan_tile_programs(n, c128, g)
    w2, i2 = sim.sim_plan_tile_programs(n, c128, g, t)
    assert np.all(info[:, 2] == t) and np.array_equal(words, w2) and np.array_equal(info, i2)
    ops, oi = sim.sim_plan_staged_ops(n, c128, g)
    assert np.all(oi[:, 2] == t)
    for tile in (0, t):
        d = sim.sim_plan_describe(n, c128, g, sim.plan_opts("staged", tile_qubits=tile))
        assert d[0] == len(info)
        if tile:
            assert d[1:3] == last[1:3] and np.array_equal(d[3], last[3])
        last = d


@pytest.mark.parametrize("masked,tile", [(12, 13), (13, 12)])
@pytest.mark.parametrize("n", [23, 26])
@pytest.mark.parametrize("kind", ["controlled", "phase"])
def test_masked_gates_take_smaller_tiles(kind, n, masked, tile):
    """More than an eighth of a large register's gates; swaps are renamed and count only
    as the exchanges of places that are left of them."""
    from paper_1805_00988_gb300 import sim
    m = (C.gate("ry", 3, controls=(5,), params=(0.4,)) if kind == "controlled" else
         C.gate("p", 3, controls=(5, 9), params=(0.4,)))
    g = C.concat([C.gate("h", q % n) for q in range(96 - masked)] + [m] * masked + [C.gate("swap", 0, target2=9)] * 2)
    sg = sim.to_sim_gates(g)
    assert np.all(sim.sim_plan_tile_programs(n, 0, sg)[1][:, 2] == tile)
    assert np.all(sim.sim_plan_staged_ops(n, 0, sg)[1][:, 2] == tile)


# ------------------------------------------------------------------ GPU

@pytest.fixture(scope="module")
def gsim():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import sim as S
    return S


@pytest.mark.gpu
@pytest.mark.parametrize("dt,n,plan,kw", [("c64", 14, "staged", {}), ("c64", 20, "staged", {}), ("c128", 20, "staged", {}),
                                          ("c64", 24, "fused", {"fuse_k": 6}), ("c64", 26, "fused", {"fuse_k": 6}),
                                          ("c128", 21, "fused", {"fuse_k": 4}), ("c128", 22, "fused", {"fuse_k": 4})])
def test_described_passes_are_those_launched(gsim, dt, n, plan, kw):
    g = C.concat([C.haar_cz(n, 8, seed=1), C.qft(n), C.qft(n), C.gate("swap", 1, target2=n - 2)])
    passes, blocks = gsim.sim_plan_describe(n, 1 if dt == "c128" else 0, gsim.to_sim_gates(g), gsim.plan_opts(plan, **kw))[:2]
    st = gsim.State(n, dt)
    gsim.sim_profile_enable(st.h, True)
    st.apply(g, plan=plan, **kw)
    count = {k: v[0] for k, v in gsim.sim_profile_read(st.h).items()}
    st.close()
    tiles = count.get("staged", 0)
    fused = sum(v for k, v in count.items() if k.startswith("fused"))
    assert tiles + fused == passes
    if plan == "fused":
        assert fused == blocks and (tiles > 0) == (n >= (22 if dt == "c128" else 26))
