"""The stage-level weight kernels at the edges of their launch rules: the
normalisation spread over the GPU against the single-CTA kernel (which still
serves weights written over their log-weights) and the oracle, and systematic
resampling where single particles own output ranges of every length."""
import numpy as np
import pytest

from gpu_util import dev, need_gpu, ptr, stream, torch  # noqa: F401
import oracle
import paper_2504_02627_gb300 as g

pytestmark = pytest.mark.gpu


def _normalise(lw, in_place):
    lw_d = dev(lw)
    W = lw_d if in_place else torch.empty_like(lw_d)
    sc = torch.empty(2, dtype=torch.float64, device="cuda")
    g.check(g.lib().smc_k_normalise(ptr(lw_d), lw.size, ptr(W), ptr(sc), ptr(sc) + 8, stream()), "normalise")
    torch.cuda.synchronize()
    return W.cpu().numpy(), *sc.cpu().numpy()


@pytest.mark.parametrize("N", [1, 256, 257, 511, 512, 513, 152 * 512, 152 * 512 + 1, 304 * 256 + 1, 100003])
@pytest.mark.parametrize("special", ["none", "-inf", "all -inf", "nan", "+inf", "one share -inf"])
def test_normalise_over_the_gpu_matches_one_cta(N, special):
    """Both forms round the same exact sums, of at most N terms added in trees
    or in chains of N / 1024: relative error of the sum below 1e-13, of lse
    below 1e-13 + its own rounding at |lse| < 1024 (1.1e-13), so W and the ESS
    agree to 1e-12."""
    need_gpu()
    lw = 3.0 * np.random.default_rng(N).standard_normal(N) - 300.0
    if special == "-inf":
        lw[::3] = -np.inf
        lw[-1] = -301.0
    elif special == "all -inf":
        lw[:] = -np.inf
    elif special == "nan":
        lw[N // 2] = np.nan
    elif special == "+inf":
        lw[N // 2] = np.inf
    elif special == "one share -inf":
        lw[:N // 2] = -np.inf
    W, lse, ess = _normalise(lw, False)
    W1, lse1, ess1 = _normalise(lw, True)
    np.testing.assert_allclose(W, W1, rtol=1e-12, atol=0.0, equal_nan=True)
    np.testing.assert_allclose([lse, ess], [lse1, ess1], rtol=1e-12, equal_nan=True)
    if special in ("none", "-inf"):
        lse_o, ess_o, W_o = oracle.normalise(lw)
        np.testing.assert_allclose(W, W_o, rtol=1e-12, atol=0.0)
        np.testing.assert_allclose([lse, ess], [lse_o, ess_o], rtol=1e-12)


@pytest.mark.parametrize("N", [1, 255, 2048, 2049, 70001, 4194304, 4300001])
@pytest.mark.parametrize("kind", ["one", "few", "heavy", "even"])
def test_resampling_long_and_short_ranges_bit_exact(N, kind):
    """Ranges of one slot, of a warp's, of a CTA's and of all N slots; the last
    size is past the tiles whose totals every CTA adds up."""
    need_gpu()
    rng = np.random.default_rng(N)
    W = np.zeros(N)
    if kind == "one":
        W[N // 3] = 1.0
    elif kind == "few":
        W[rng.integers(0, N, size=7)] = rng.uniform(0.1, 1.0, size=7)
    elif kind == "heavy":
        W = rng.gamma(0.05, size=N) + 1e-300
    else:
        W[:] = 1.0
    W /= W.sum()
    r64 = 0xD1B54A32D192ED03
    W_d = dev(W)
    q = torch.empty(N, dtype=torch.int64, device="cuda")
    anc = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    st = torch.full((1,), 99, dtype=torch.int32, device="cuda")
    scr = torch.full((g.lib().smc_k_resample_scratch_bytes(N),), 255, dtype=torch.uint8, device="cuda")
    g.check(g.lib().smc_k_resample(ptr(W_d), N, r64, ptr(q), ptr(anc), ptr(st), ptr(scr), stream()), "resample")
    torch.cuda.synchronize()
    _, q_o = oracle.quantise(W)
    _, a_o = oracle.systematic(q_o, r64)
    assert int(st.cpu()[0]) == 0
    np.testing.assert_array_equal(q.cpu().numpy().astype(np.uint64), np.asarray(q_o).astype(np.uint64))
    np.testing.assert_array_equal(anc.cpu().numpy(), a_o)
