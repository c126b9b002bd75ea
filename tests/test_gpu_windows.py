"""Step counts around the ends of the coefficient table's window in shared memory (32
rows in FP32, 16 in FP64, two of them in flight), in every step loop, against the
counting launch, which reads the table in place.  The counting launch finds buffers
that no other launch of its shape has written."""
import numpy as np
import pytest
import torch

from paper_2410_08267_gb300 import nuprof as nu
from paper_2410_08267_gb300 import workloads as W

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
PLAIN = W.plain_small(precision=W.MIXED)[0].replace(radii=np.geomspace(1.0, 3000.0, 12), n_q=30, n_mu=12)


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


def _run_and_count(pb):
    """Momenta and results of a normal run, and of a counting launch after the device
    memory was put back to what it was before the run and the results were overwritten
    by a run of another tile, which adds in another order."""
    held = []

    @nu.ALLOC_FN
    def alloc(nbytes, ctx):
        held.append(torch.zeros(nbytes, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        return held[-1].data_ptr()

    @nu.FREE_FN
    def free(ptr, nbytes, ctx):
        pass

    cosmo, halo, relic, radii, grid, opts = nu.structs(pb, flags=nu.NU_FLAG_KEEP_QI)
    opts.alloc, opts.free = alloc, free
    h = nu.nu_profile_create(cosmo, halo, relic, radii, grid, opts)
    other = nu.nu_opts()
    other.block, other.tpt = 96, 1
    b, b_other = nu.nu_batch_create([h]), nu.nu_batch_create([h], other)
    try:
        before = held[0].clone()
        nu.nu_batch_run(b)
        want = (nu.nu_profile_qi(h, pb.n_traj), *nu.nu_profile_result(h, pb.n_out))
        nu.nu_batch_run(b_other)
        overwritten = nu.nu_profile_result(h, pb.n_out)[0]
        held[0].copy_(before)
        torch.cuda.synchronize()
        assert not nu.nu_profile_qi(h, pb.n_traj).any()
        nu.nu_batch_branch_counts(b)
        got = (nu.nu_profile_qi(h, pb.n_traj), *nu.nu_profile_result(h, pb.n_out))
        return want, got, overwritten
    finally:
        nu.nu_batch_destroy(b)
        nu.nu_batch_destroy(b_other)
        nu.nu_profile_destroy(h)


@pytest.mark.parametrize("n_steps", [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 96, 97])
@pytest.mark.parametrize("loop", [{}, {"masses": (0.05, 0.1, 0.2)}, {"radii": np.geomspace(1.0, 3000.0, 800)},
                                  {"precision": W.FP64},
                                  {"precision": W.FP64, "radii": np.geomspace(1.0, 3000.0, 60)}],
                         ids=["one_a_lane", "masses", "two_a_lane", "fp64_split", "fp64"])
def test_window_ends_are_bitwise_the_counting_loop(loop, n_steps):
    want, got, overwritten = _run_and_count(PLAIN.replace(n_steps=n_steps, **loop))
    assert np.any(overwritten != want[1])
    for x, y in zip(want, got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("loop", [{}, {"radii": np.geomspace(1.0, 3000.0, 800)}, {"precision": W.FP64}],
                         ids=["one_a_lane", "two_a_lane", "fp64"])
def test_longest_runs_are_bitwise_the_counting_loop(loop):
    want, got, _ = _run_and_count(PLAIN.replace(n_steps=nu.NU_MAX_STEPS, **loop))
    for x, y in zip(want, got):
        assert np.array_equal(x, y)
