"""Stage-level moves in the order of their step counts, beside other work: the
results are those of the particles' own order bit for bit, whichever route a
call takes.  Which call takes which route: test_host_ordered_moves.py."""
import numpy as np
import pytest

from gpu_util import dev, need_gpu, ptr, torch  # noqa: F401
from paper_2504_02627_gb300 import _binding as B

pytestmark = pytest.mark.gpu
D, N = 100, 6007
# (kind, dimensions, observations, particles, precision) of moves that are ordered
# (test_host_ordered_moves.py holds them against the rule); 97 particles are not
ORDERED = [("gauss", D, 0, N, 0), ("gauss", D, 0, 9800, 0), ("gauss", D, 0, N, 1), ("gauss", D, 0, N, 2),
           ("gauss", 80, 0, 16411, 2), ("gauss", 40, 0, 20011, 0), ("logistic", 25, 1000, 2500, 0), ("logistic", 40, 64, 9800, 0)]


def model(kind, D, n):
    rng = np.random.default_rng(D)
    if kind == "logistic":
        return B.ModelData(B.LOGISTIC, D, n, X=rng.standard_normal((n, D)), y=(rng.uniform(size=n) < 0.5), hyper=(1.0,))
    A = rng.standard_normal((D, D))
    return B.ModelData(B.GAUSS_DENSE, D, mu=rng.standard_normal(D), prec=A @ A.T / D + np.eye(D))


def _state(seed, n=N, D=D):
    t = torch.Generator(device="cuda").manual_seed(seed)
    x = [torch.randn(D, n, device="cuda", generator=t) for _ in range(3)]
    return x + [torch.zeros(n, dtype=torch.float64, device="cuda")]


def _move(dm, x, S, s, precision=0):
    n = x[3].numel()
    B.check(B.lib().smc_k_leapfrog(dm.h, *map(ptr, x), ptr(S), 0.01, n, n, precision, s.cuda_stream), "leapfrog")


def test_moves_beside_captures_and_busy_streams():
    need_gpu()
    a, b, c = (torch.cuda.Stream() for _ in range(3))
    dm = B.DevModel(model("gauss", D, 0), a.cuda_stream)
    S = dev(np.random.default_rng(1).integers(0, 40, size=N).astype(np.int32))
    x = [[t.clone() for t in _state(2)] for _ in range(4)]
    big, S_big = _state(3, 262144), torch.full((262144,), 60, dtype=torch.int32, device="cuda")
    y = torch.zeros(1024, device="cuda")
    torch.cuda.synchronize()
    _move(dm, x[0], S, a)                            # ordered
    with torch.cuda.stream(a):
        y.add_(1)                                    # kernels that the capture below will need
    torch.cuda.synchronize()
    # another stream's capture in the global mode, with the room last used on
    # a third stream: the capture goes through
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=c, capture_error_mode="global"):
        y.add_(1)
        _move(dm, x[1], S, b)
        y.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert float(y[0]) == 3.0
    # the room is busy on another stream
    _move(dm, big, S_big, a)
    _move(dm, x[2], S, b)
    torch.cuda.synchronize()
    # the move itself captured, and replayed
    keep = [t.clone() for t in _state(2)]
    graph2 = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph2, stream=c):
        _move(dm, x[3], S, c)
    for t in (0, 1):
        for i in range(4):
            x[3][i].copy_(keep[i])
        graph2.replay()
        torch.cuda.synchronize()
        for k in (1, 2, 3):
            for u, v in zip(x[0], x[k]):
                assert torch.equal(u, v)
    dm.close()


@pytest.mark.parametrize("kind,dim,obs,n,precision", ORDERED)
def test_ordered_moves_of_every_kind(kind, dim, obs, n, precision):
    """Ragged, equal and zero step counts, against the same particles in
    launches of 97, which are not ordered.  The gradients are not those of the
    positions: a particle without steps keeps the one it came with."""
    need_gpu()
    s = torch.cuda.current_stream()
    dm = B.DevModel(model(kind, dim, obs), s.cuda_stream)
    start = _state(n, n, dim)
    rng = np.random.default_rng(n)
    for counts in (rng.integers(0, 9, size=n), np.full(n, 3), rng.integers(0, 2000, size=n) // 400, np.zeros(n, int)):
        S = dev(counts.astype(np.int32))
        whole = [t.clone() for t in start]
        _move(dm, whole, S, s, precision)
        for lo in range(0, n, 97):
            part = [t[..., lo:lo + 97].clone(memory_format=torch.contiguous_format) for t in start]
            _move(dm, part, S[lo:lo + 97].clone(), s, precision)
            for u, v in zip(part, whole):
                assert torch.equal(u, v[..., lo:lo + 97])
        still = S == 0
        assert torch.equal(whole[2][:, still], start[2][:, still])
    dm.close()
