"""Sampling at the edges of its levels (8192-amplitude blocks, 256-amplitude
sub-blocks, 32-amplitude eighths; below 2^8 amplitudes one prefix): states whose
weight sits on few amplitudes, at the ends of the levels, against the FP64 oracle.

The weights are the squares of the stored amplitudes on both sides, so shots
are equal except within rounding of a prefix boundary: prefixes agree to about
1e-14 of the total, with at most 2^15 boundaries and 20000 shots that is an
expected 1e-5 shots; two are allowed.  No shot lands on a zero amplitude.
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


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 12, 13, 14, 15])
def test_shots_match_oracle(sim, orc, dt, n):
    N = 1 << n
    rng = np.random.default_rng(n)
    noise = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    ends = np.arange(N) % 32 == 31
    states = [np.where(np.arange(N) == N - 1, 1, 0), np.where(np.arange(N) == 0, 1, 0),
              np.where(ends | (np.arange(N) == 0), noise, 0), np.where(rng.random(N) < 3 / N, noise, 0),
              noise, noise * 10.0 ** rng.uniform(-12, 0, N)]
    st = sim.State(n, dt)
    for psi in states:
        psi = psi.astype(np.complex64 if dt == "c64" else np.complex128)
        if not psi.any():
            psi[N // 2] = 1
        st.load(psi)
        got = st.sample(20000, seed=3)
        ref = orc.sample(psi.astype(np.complex128), 20000, seed=3)
        assert np.count_nonzero(got != ref) <= 2
        assert np.all(psi[got] != 0)
    st.close()


def test_zero_norm_is_refused(sim):
    st = sim.State(9, "c64")
    st.load(np.zeros(512, dtype=np.complex64))
    with pytest.raises(sim.SimError):
        st.sample(10, seed=1)
    st.close()
