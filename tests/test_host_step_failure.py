"""An iteration whose launches fail part of the way.  Once its first kernel has
run, the step histogram and the weights' total hold this iteration's counts: a
second attempt would add to them and write the launch order far past its end,
so the handle refuses every further step until smc_reset, which empties them.
Run on the host's CUDA runtime: no kernel runs."""
import ctypes as C

import pytest

import host_cuda
import paper_2504_02627_gb300 as g
import workloads


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_cuda.load(tmp_path_factory.mktemp("host_cuda"))


def _handle(lib, n_particles=256):
    w = workloads.gauss10()
    md = g.ModelData.from_workload(w)
    cfg = g.make_config(seed=1, **dict(w["run"], n_particles=n_particles))
    h = C.c_void_p()
    lib.host_cuda_fail(b"", 0, 0)
    assert lib.smc_init(C.byref(h), C.byref(cfg), C.byref(md.struct), None) == 0
    host_cuda.launches(lib)
    return h


@pytest.mark.parametrize("n_particles", [256, 5000])     # resampling and order in one kernel, and in three
@pytest.mark.parametrize("kernel,profile", [(b"resample", 0), (b"traj", 0), (b"traj", 1), (b"move_stats", 0),
                                            (b"chees_finish", 0)])
def test_a_step_that_failed_is_not_tried_again(lib, n_particles, kernel, profile):
    h = _handle(lib, n_particles)
    lib.smc_profile(h, profile)
    lib.host_cuda_fail(kernel, host_cuda.NOMEM, 0)
    assert lib.smc_step(h, None) == host_cuda.E_NOMEM
    assert "k_weights_steps" in " ".join(host_cuda.launches(lib))
    lib.host_cuda_fail(b"", 0, 0)
    assert lib.smc_step(h, None) == host_cuda.E_STATE
    assert lib.smc_run(h, 4, None) == host_cuda.E_STATE
    assert host_cuda.launches(lib) == []                  # nothing that adds to the counts
    assert lib.smc_reset(h, 2) == 0
    assert lib.smc_step(h, None) == 0
    lib.smc_destroy(h)


def test_a_step_that_never_began_may_be_tried_again(lib):
    h = _handle(lib)
    lib.host_cuda_fail(b"weights_steps", host_cuda.NOMEM, 0)
    assert lib.smc_step(h, None) == host_cuda.E_NOMEM
    lib.host_cuda_fail(b"", 0, 0)
    assert lib.smc_step(h, None) == 0
    assert lib.smc_step(h, None) == 0
    # another call's error left behind in the thread: reported, nothing launched
    lib.host_cuda_leave_error(host_cuda.NOMEM)
    host_cuda.launches(lib)
    assert lib.smc_step(h, None) == host_cuda.E_NOMEM
    assert host_cuda.launches(lib) == []
    assert lib.smc_step(h, None) == 0
    assert lib.smc_step(h, None) == 0
    # a step that fails while its graph is captured has not run either
    lib.host_cuda_fail(b"traj", host_cuda.NOMEM, 0)
    assert lib.smc_run(h, 4, None) == host_cuda.E_NOMEM
    lib.host_cuda_fail(b"", 0, 0)
    host_cuda.launches(lib)
    assert lib.smc_run(h, 4, None) == 0
    assert host_cuda.launches(lib).count("graph") == 2
    lib.smc_destroy(h)


def test_a_capture_that_failed_leaves_the_buffers_in_place(lib):
    """The second of the two captured steps fails: the particles are still where
    the last step that ran left them, and the next run starts from there."""
    h = _handle(lib)
    lib.host_cuda_fail(b"move_stats", host_cuda.NOMEM, 1)
    assert lib.smc_run(h, 4, None) == host_cuda.E_NOMEM
    lib.host_cuda_fail(b"", 0, 0)
    host_cuda.launches(lib)
    assert lib.smc_run(h, 4, None) == 0
    names = host_cuda.launches(lib)
    assert names.count("graph") == 2
    assert sum("k_weights_steps" in n for n in names) == 2     # captured; none to align the buffers
    lib.smc_destroy(h)
