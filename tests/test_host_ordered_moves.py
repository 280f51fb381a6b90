"""Which stage-level moves take the launch order, and what the call does beside
other streams' work and captures, on the host's CUDA runtime (no kernel runs;
test_gpu_ordered_moves.py has the results on the GPU)."""
import ctypes as C

import numpy as np
import pytest

import host_cuda
from paper_2504_02627_gb300 import _binding as B
from test_gpu_ordered_moves import D, ORDERED, model


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_cuda.load(tmp_path_factory.mktemp("host_cuda"))


def _model(lib, md=None):
    md = md or model("gauss", D, 0)
    m = C.c_void_p()
    assert lib.smc_model_create(C.byref(m), C.byref(md.struct), None) == 0
    host_cuda.launches(lib)
    return m


def _ordered(lib, m, stream, N=6007, precision=0):
    """Whether a move on this stream was ordered."""
    room = C.c_void_p(4096)                       # never read: no kernel runs
    assert lib.smc_k_leapfrog(m, room, room, room, room, room, 0.1, N, N, precision, C.c_void_p(stream)) == 0
    names = host_cuda.launches(lib)
    assert any("traj" in n for n in names)
    return any("k_order_steps" in n for n in names)


def test_a_capture_of_another_thread_is_left_whole(lib):
    m = _model(lib)
    lib.host_cuda_foreign_capture(0)
    assert _ordered(lib, m, 16)
    lib.host_cuda_foreign_capture(1)
    assert _ordered(lib, m, 32)                   # the room's last move ran on another stream, and has ended
    assert not lib.host_cuda_foreign_capture_broken()
    lib.host_cuda_foreign_capture(0)
    assert lib.host_cuda_mode() == 0              # as the thread had it: global
    lib.smc_model_destroy(m)


def test_a_move_without_the_room_runs_in_the_particles_order(lib):
    m = _model(lib)
    assert _ordered(lib, m, 16)
    lib.host_cuda_event_busy(1)
    assert _ordered(lib, m, 16)                   # behind its own stream's move
    assert not _ordered(lib, m, 32)               # that move may still read the room
    lib.host_cuda_event_busy(0)
    assert _ordered(lib, m, 32)
    lib.host_cuda_capture(1)
    assert not _ordered(lib, m, 32)               # a replay could overlap later calls
    lib.host_cuda_capture(0)
    assert lib.host_cuda_last_error() == 0        # the busy event is no error of the caller's
    lib.smc_model_destroy(m)


def test_a_model_outlives_the_moves_that_use_its_room(lib):
    """The room is given back behind the last move that writes it, on whatever
    stream that ran."""
    m = _model(lib)
    lib.smc_model_destroy(m)
    assert host_cuda.launches(lib) == []
    m = _model(lib)
    assert _ordered(lib, m, 32)
    lib.smc_model_destroy(m)
    assert host_cuda.launches(lib) == ["wait"]


def test_a_move_whose_order_fails_still_runs(lib):
    m = _model(lib)
    lib.host_cuda_fail(b"k_order_steps", host_cuda.NOMEM, 0)
    assert not _ordered(lib, m, 16)
    assert lib.host_cuda_last_error() == 0
    lib.host_cuda_fail(b"", 0, 0)
    # an error that an earlier call left behind is not taken for the order's
    lib.host_cuda_leave_error(host_cuda.NOMEM)
    assert not _ordered(lib, m, 16)
    assert lib.host_cuda_last_error() == host_cuda.NOMEM
    lib.host_cuda_leave_error(0)
    lib.smc_model_destroy(m)


@pytest.mark.parametrize("kind,dim,obs,n,precision", ORDERED)
def test_the_gpu_tests_cases_are_ordered(lib, kind, dim, obs, n, precision):
    m = _model(lib, model(kind, dim, obs))
    assert _ordered(lib, m, 16, n, precision)
    assert not _ordered(lib, m, 16, 97, precision)
    lib.smc_model_destroy(m)


@pytest.mark.parametrize("kind,dim,obs,n,precision", [
    ("gauss", 100, 0, 8192, 0), ("gauss", 64, 0, 9728, 0),                      # 152 tiles of 64 at most
    ("logistic", 25, 1000, 2432, 0), ("logistic", 64, 300, 4096, 0),            # of 16, of 64 (streamed)
    ("gauss", 64, 0, 40000, 1), ("gauss", 32, 0, 30000, 0),                      # the gather costs what it saves; no tiles
])
def test_moves_that_ordering_makes_slower_are_not_ordered(lib, kind, dim, obs, n, precision):
    m = _model(lib, model(kind, dim, obs))
    assert not _ordered(lib, m, 16, n, precision)
    lib.smc_model_destroy(m)


def test_only_models_whose_moves_are_ordered_keep_room_for_the_order(lib):
    rng = np.random.default_rng(0)
    def room(md):
        m = C.c_void_p()
        before = lib.host_cuda_allocated()
        assert lib.smc_model_create(C.byref(m), C.byref(md.struct), None) == 0
        lib.smc_model_destroy(m)
        return lib.host_cuda_allocated() - before
    gauss = lambda D: B.ModelData(B.GAUSS_DENSE, D, mu=np.zeros(D), prec=np.eye(D))
    assert room(B.ModelData(B.BANANA, 50, hyper=(10.0, 0.1))) < 1 << 16
    assert room(gauss(32)) < 1 << 16                  # never ordered, at any particle count
    assert room(gauss(33)) > 1 << 20
    assert room(B.ModelData(B.LOGISTIC, 25, 1000, X=rng.standard_normal((1000, 25)), y=np.zeros(1000),
                            hyper=(1.0,))) > 1 << 20
