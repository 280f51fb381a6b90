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
