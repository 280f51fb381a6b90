"""The FP32 launches that a rule on sizes chooses between give the same bits on
either side of every line: gradients, log densities and moves of the first
particles of a large launch against a launch of those alone."""
import numpy as np
import pytest

from gpu_util import dev, need_gpu, ptr, stream, torch  # noqa: F401
from paper_2504_02627_gb300 import _binding as B
from test_gpu_split import _move, _same_bits

pytestmark = pytest.mark.gpu


def _gauss(D, mu=None):
    rng = np.random.default_rng(D)
    A = rng.standard_normal((D, D))
    mu = rng.standard_normal(D) if mu is None else mu
    return B.DevModel(B.ModelData(B.GAUSS_DENSE, D, mu=mu, prec=A @ A.T / D + np.eye(D), c=0.7), stream())


def _check(dm, D, n, larger, eps):
    g = torch.Generator(device="cuda").manual_seed(D)
    big = max(larger)
    th, p = (torch.randn(D, big, device="cuda", generator=g) for _ in range(2))
    S = dev(np.random.default_rng(D).integers(0, 7, size=big).astype(np.int32))
    small = _move(dm, th, p, S, eps, n)
    for N in larger:
        _same_bits(small, _move(dm, th, p, S, eps, N), n)
    dm.close()


@pytest.mark.parametrize("D", [33, 47, 48, 49, 63, 64, 65, 96, 97, 128])
def test_dense_gaussian_tiles(D):
    need_gpu()
    _check(_gauss(D), D, 61, (3071, 3072, 6143, 6144, 6205), 0.02)


@pytest.mark.parametrize("D", [5, 7, 8, 9, 15, 16, 17, 31, 32])
def test_gaussian_rows_and_particles(D):
    """Moves: 32768 particles up to 16 dimensions, else 1245184 values; gradients
    alone: 131072 lanes."""
    need_gpu()
    lanes = 8 if D <= 8 else 16 if D <= 16 else 32
    move = 32768 if D <= 16 else 1245184 // D
    _check(_gauss(D), D, 301, (131072 // lanes, 131072 // lanes + 1, move, move + 1), 0.02)


@pytest.mark.parametrize("G", [15, 20, 32, 50, 51, 62])
def test_hierarchical_normal_register_caps(G):
    """Two CTAs of 128 particles an SM, and more."""
    need_gpu()
    rng = np.random.default_rng(G)
    md = B.ModelData(B.HIER_NORMAL, G + 2, G, group_mean=rng.standard_normal(G), group_n=np.full(G, 20.0),
                     group_ss=np.full(G, 19.0), hyper=(1.0,))
    few = 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    _check(B.DevModel(md, stream()), G + 2, 301, (few, few + 1), 0.01)


def test_rows_of_a_diverged_particle():
    """Deviations that overflow stay infinite where the row sums do: the lanes past
    D add nothing to them (5 of 8 lanes; all elements of P positive)."""
    need_gpu()
    D = 5
    mu = np.zeros(D)
    mu[0] = -3e38
    dm = B.DevModel(B.ModelData(B.GAUSS_DENSE, D, mu=mu, prec=0.5 * np.eye(D) + 0.5), stream())
    th = torch.zeros(D, 1, device="cuda")
    th[0] = 3e38                                   # the deviation is infinite, the position is not
    p, gr, lp = torch.zeros_like(th), torch.zeros_like(th), torch.zeros(1, dtype=torch.float64, device="cuda")
    S = dev(np.array([2], np.int32))
    B.check(B.lib().smc_k_leapfrog(dm.h, ptr(th), ptr(p), ptr(gr), ptr(lp), ptr(S), 0.1, 1, 1, 0, stream()), "leapfrog")
    torch.cuda.synchronize()
    assert torch.all(th == -np.inf) and torch.all(gr == np.inf)
    dm.close()
