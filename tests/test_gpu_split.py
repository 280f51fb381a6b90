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


@pytest.mark.parametrize("D", [2, 4, 8, 16, 18, 64])
def test_banana_log_density_is_its_written_fp32_form(D):
    """The FP32 terms to the last bit (an FMA of FP32 values is exact in FP64 but
    for its rounding), their FP64 sum up to its order."""
    need_gpu()
    dm = B.DevModel(B.ModelData(B.BANANA, D, hyper=(10.0, 0.1)), stream())
    n = 500
    th = torch.as_tensor(np.random.default_rng(D).standard_normal((D, n)).astype(np.float32)).cuda()
    gr, lp = torch.zeros(D, n, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    B.check(B.lib().smc_k_target(dm.h, ptr(th), n, n, ptr(lp), ptr(gr), 0, stream()), "target")
    f = np.float32
    fma = lambda x, y, z: (x.astype(np.float64) * y.astype(np.float64) + z.astype(np.float64)).astype(f)
    xo, xe = th.cpu().numpy()[0::2], th.cpu().numpy()[1::2]
    full = lambda v: np.full_like(xo, f(v))
    u = fma(full(-0.1), fma(xo, xo, full(-10.0)), xe)
    s, t = f(-0.05) * xo, f(0.5) * u
    terms = fma(-t, u, s * xo) if D == 2 else fma(s, xo, -(t * u))
    want = terms.astype(np.float64).sum(axis=0)
    got = lp.cpu().numpy()
    const = np.median(got - want)                       # the normalising constant
    assert np.all(np.abs(got - want - const) <= 1e-13 * (np.abs(terms).sum(axis=0) + abs(const)))
    dm.close()


@pytest.mark.parametrize("kind,D,n,N", [("gauss", 100, 0, 3100), ("gauss", 40, 0, 20011), ("logistic", 25, 1000, 515),
                                        ("logistic", 40, 3000, 130)])
@pytest.mark.parametrize("precision", [0, 1])
def test_ordered_moves_give_the_bits_of_unordered_ones(kind, D, n, N, precision):
    """Launches above the ordering threshold against the same particles in
    launches of 97 (below it): ragged, equal and zero step counts, on two
    streams in turn."""
    need_gpu()
    if kind == "logistic" and precision:
        pytest.skip("the regressions are ordered in FP32 only")
    rng = np.random.default_rng(N)
    if kind == "gauss":
        A = rng.standard_normal((D, D))
        md = B.ModelData(B.GAUSS_DENSE, D, mu=rng.standard_normal(D), prec=A @ A.T / D + np.eye(D))
    else:
        md = B.ModelData(B.LOGISTIC, D, n, X=rng.standard_normal((n, D)), y=(rng.uniform(size=n) < 0.5), hyper=(1.0,))
    dm = B.DevModel(md, stream())
    th, p, gr = (torch.randn(D, N, device="cuda") for _ in range(3))
    lp = torch.randn(N, dtype=torch.float64, device="cuda")
    other = torch.cuda.Stream()
    for turn, S in enumerate((rng.integers(0, 9, size=N), np.full(N, 3), rng.integers(0, 2000, size=N) // 400)):
        S_d = dev(S.astype(np.int32))
        torch.cuda.synchronize()
        whole = [x.clone() for x in (th, p, gr, lp)]
        torch.cuda.synchronize()
        s = other.cuda_stream if turn == 1 else stream()
        B.check(B.lib().smc_k_leapfrog(dm.h, *map(ptr, whole), ptr(S_d), 0.01, N, N, precision, s), "leapfrog")
        torch.cuda.synchronize()
        for lo in range(0, N, 97):
            hi = min(N, lo + 97)
            part = [x[..., lo:hi].clone(memory_format=torch.contiguous_format) for x in (th, p, gr, lp)]
            Sp = S_d[lo:hi].clone()
            B.check(B.lib().smc_k_leapfrog(dm.h, *map(ptr, part), ptr(Sp), 0.01, hi - lo, hi - lo, precision, stream()),
                    "leapfrog")
            for a, b in zip(part, whole):
                assert torch.equal(a, b[..., lo:hi])
    dm.close()
