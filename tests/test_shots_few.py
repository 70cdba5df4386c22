"""Sampling on both sides of the line where the pass over the state writes the sums of
its 32-amplitude eighths (one shot in 2048 amplitudes complex64, in 4096 complex128):
states whose weight sits on few amplitudes, at the ends of the levels, against the
FP64 oracle.  As in test_shots.py, shots are equal except within rounding of a prefix boundary:
prefixes agree to about 1e-14 of the total, with 2^20 boundaries and 5000 shots a state that is
an expected 1e-4 shots; one is allowed.  No shot lands on a zero amplitude.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1805_00988_gb300 import sim as s
    return s


@pytest.mark.parametrize("dt,n,shots", [("c64", 14, 7), ("c64", 20, 1), ("c64", 20, 511), ("c64", 20, 512), ("c128", 17, 31),
                                        ("c128", 20, 255), ("c128", 20, 256)])
def test_few_shots_match_oracle(sim, orc, dt, n, shots):
    N = 1 << n
    rng = np.random.default_rng(n)
    noise = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    ends = np.arange(N) % 32 == 31
    states = [np.where(np.arange(N) == N - 1, 1, 0), np.where(np.arange(N) == 0, 1, 0), np.where(ends, noise, 0),
              np.where(rng.random(N) < 3 / N, noise, 0), noise, noise * 10.0 ** rng.uniform(-12, 0, N)]
    st = sim.State(n, dt)
    for psi in states:
        psi = psi.astype(np.complex64 if dt == "c64" else np.complex128)
        if not psi.any():
            psi[N // 2] = 1
        st.load(psi)
        off = 0
        for seed in range(10):
            got = st.sample(shots, seed=seed)
            off += np.count_nonzero(got != orc.sample(psi.astype(np.complex128), shots, seed=seed))
            assert np.all(psi[got] != 0)
            if dt == "c64":
                again, norm, _ = sim.sim_sample_observe(st.h, shots, seed)
                assert np.array_equal(again, got) and norm > 0
        assert off <= 1
    st.close()
