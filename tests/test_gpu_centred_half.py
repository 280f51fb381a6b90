"""The centred trajectories with two CTAs to an SM (many particles, D <= 64, short
passes): positions, momenta, the end-point gradient and log pi of sampled
particles against the oracle, with the bounds of test_gpu_centred, at every
operand width (16, 32, 48 and 64 dimensions, the last with three copy stages),
one observation tile and several, ragged last tiles, and every place in a tile."""
import numpy as np
import pytest

from gpu_util import dev, f32r, need_gpu, oracle_target, ptr, rounded_workload, stream, torch  # noqa: F401
from test_gpu_centred import PREC, _dev_state, _log_scale, _theta, centred_bound
import oracle
import paper_2504_02627_gb300 as g
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,eps", [
    (lambda: workloads.logistic(), 1e-3),                          # 8 tiles, D = 25
    (lambda: workloads.logistic(n=100, d_features=6), 2e-3),       # one tile, D = 7
    (lambda: workloads.linear_gauss(n=200, D=6), 0.005),
    (lambda: workloads.logistic_large(n=700, D=40), 2e-3),
    (lambda: workloads.logistic_large(n=1153, D=64), 2e-3),
    (lambda: workloads.logistic(n=1700), 1e-3),                    # 14 tiles: past the rule, 128 particles per CTA
])
def test_two_ctas_per_sm_against_the_oracle(make, eps):
    need_gpu()
    w = rounded_workload(make())
    t = oracle_target(w)
    dm = g.DevModel(g.ModelData.from_workload(w), stream())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N = 128 * sms + 19                               # more tiles than SMs: no cluster
    ld = N + 13
    th = _theta(w, N, seed=5)
    p = f32r(np.random.default_rng(9).standard_normal((N, w["D"])))
    S = np.random.default_rng(10).integers(0, 7, N).astype(np.int32)
    t_d, p_d = _dev_state(th, ld), _dev_state(p, ld)
    g_d = torch.zeros_like(t_d)
    lp_d = torch.zeros(ld, dtype=torch.float64, device="cuda")
    lib = g.lib()
    g.check(lib.smc_k_target(dm.h, ptr(t_d), N, ld, ptr(lp_d), ptr(g_d), PREC, stream()), "target")
    g.check(lib.smc_k_leapfrog(dm.h, ptr(t_d), ptr(p_d), ptr(g_d), ptr(lp_d), ptr(dev(S)), eps, N, ld, PREC,
                               stream()), "leapfrog")
    # every row of the first tile, the last tile's, and some between
    idx = np.unique(np.concatenate([np.arange(128), np.arange(N - 19, N), np.random.default_rng(2).choice(N, 32)]))
    th_g, p_g, gr_g = (x.cpu().numpy()[:, idx].T.astype(np.float64) for x in (t_d, p_d, g_d))
    lp_g = lp_d.cpu().numpy()[idx]
    th_o, p_o, _, _ = oracle.leapfrog(t, th[idx], p[idx], eps, S[idx])
    c = th.mean(axis=0)
    dg = np.maximum(centred_bound(w, th[idx], c), centred_bound(w, th_o, c))
    Sc = S[idx][:, None].astype(np.float64)
    rms = lambda a: np.sqrt(np.mean(a**2))
    assert np.all(np.abs(p_g - p_o) <= (Sc + 1) * eps * dg + 1e-5 * Sc * (np.abs(p_o) + rms(p_o)))
    assert np.all(np.abs(th_g - th_o) <= Sc**2 * eps**2 * dg + 1e-5 * Sc * (np.abs(th_o) + rms(th_o)))
    lp_at, gr_at = oracle.logpi(t, th_g)
    assert np.all(np.abs(lp_g - lp_at) <= 1e-5 * _log_scale(w, th_g))
    assert np.all(np.abs(gr_g - gr_at) <= centred_bound(w, th_g, c) + 1e-4 * np.abs(gr_at))
    dm.close()
