"""The kernels that spread a particle over several threads (the dense Gaussian by
rows, the banana by pairs): every sum keeps the order of a thread that holds
the whole particle, so a launch small enough for the row kernel gives the bits
of one that takes a thread per particle, and a banana's particles give the
same bits whatever shares their warp."""
import numpy as np
import pytest

from gpu_util import dev, need_gpu, ptr, stream, torch  # noqa: F401
import paper_2504_02627_gb300 as g
from paper_2504_02627_gb300 import _binding as B

pytestmark = pytest.mark.gpu


def _move(dm, th, p, S, eps, N):
    D = th.shape[0]
    t = [x[:, :N].clone(memory_format=torch.contiguous_format) for x in (th, p)]   # moved in place
    gr = torch.zeros(D, N, device="cuda")
    lp = torch.zeros(N, dtype=torch.float64, device="cuda")
    lib = B.lib()
    B.check(lib.smc_k_target(dm.h, ptr(t[0]), N, N, ptr(lp), ptr(gr), 0, stream()), "target")
    first = [gr.clone(), lp.clone()]
    s = S[:N].contiguous()
    B.check(lib.smc_k_leapfrog(dm.h, ptr(t[0]), ptr(t[1]), ptr(gr), ptr(lp), ptr(s), eps, N, N, 0, stream()),
            "leapfrog")
    torch.cuda.synchronize()
    return first + t + [gr, lp]


def _same_bits(small, large, n):
    for a, b in zip(small, large):
        assert torch.equal(a[..., :n], b[..., :n])


@pytest.mark.parametrize("D", [5, 8, 9, 16, 17, 32])
def test_gaussian_rows_give_the_bits_of_a_thread_per_particle(D):
    need_gpu()
    rng = np.random.default_rng(D)
    A = rng.standard_normal((D, D))
    dm = B.DevModel(B.ModelData(B.GAUSS_DENSE, D, mu=rng.standard_normal(D), prec=A @ A.T / D + np.eye(D), c=0.7),
                    stream())
    n, big = 301, 152 * 2048 * 4 // D + 1        # the row kernel's particle limit, exceeded
    th = torch.randn(D, big, device="cuda")
    p = torch.randn(D, big, device="cuda")
    S = dev(rng.integers(0, 9, size=big).astype(np.int32))
    small, large = _move(dm, th, p, S, 0.05, n), _move(dm, th, p, S, 0.05, big)
    _same_bits(small, large, n)
    dm.close()


@pytest.mark.parametrize("D", [2, 6, 16, 18, 34, 50, 64])
def test_banana_pairs_are_independent_of_their_neighbours(D):
    need_gpu()
    rng = np.random.default_rng(D)
    dm = B.DevModel(B.ModelData(B.BANANA, D, hyper=(10.0, 0.1)), stream())
    n = 333
    th = torch.randn(D, n, device="cuda")
    p = torch.randn(D, n, device="cuda")
    S = dev(rng.integers(0, 20, size=n).astype(np.int32))
    whole = _move(dm, th, p, S, 0.02, n)
    for i in (0, 31, 32, 332):                       # one particle at a time, and the ragged end
        one = _move(dm, th[:, i:i + 1], p[:, i:i + 1], S[i:i + 1], 0.02, 1)
        for a, b in zip(one, whole):
            assert torch.equal(a[..., 0], b[..., i])
    dm.close()
