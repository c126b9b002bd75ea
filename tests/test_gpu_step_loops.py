"""Every step loop of the trajectory kernel against the counting launch, which
integrates each trajectory alone with the general force (every branch tested
per lane, no vote): the same n/nbar, error estimate and q_i, bit for bit."""
import numpy as np
import pytest

from paper_2410_08267_gb300 import nuprof as nu
from paper_2410_08267_gb300 import workloads as W

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


def _both(pb, block, tpt):
    """Results of a normal run and of the counting run of one request."""
    h = nu.create(pb, block=block, tpt=tpt, flags=nu.NU_FLAG_KEEP_QI)
    b = nu.nu_batch_create([h])
    try:
        nu.nu_batch_run(b)
        runs = [(*nu.nu_profile_result(h, pb.n_out), nu.nu_profile_qi(h, pb.n_traj))]
        nu.nu_batch_branch_counts(b)
        runs.append((*nu.nu_profile_result(h, pb.n_out), nu.nu_profile_qi(h, pb.n_traj)))
        return runs
    finally:
        nu.nu_batch_destroy(b)
        nu.nu_profile_destroy(h)


PLAIN = W.plain_small(precision=W.MIXED)[0]
CASES = {
    # whole warps that stay in the NFW part, leave it and come back
    "core_and_edge": PLAIN.replace(radii=np.geomspace(1.0, 3000.0, 7), n_steps=203),
    "wide_fit_edge_at_its_end": PLAIN.replace(c=16.0, n_steps=120),
    "narrow_fit_edge_at_its_end": PLAIN.replace(c=8.0, n_steps=120),
    "logarithm_above_16": PLAIN.replace(c=25.0, n_steps=120),
    "edge_below_one": PLAIN.replace(c=0.5, n_steps=120),
    # the NFW edge lies beyond R before the onset: the bounds of the stages differ
    "past_the_onset": PLAIN.replace(z_end=6.0, n_steps=150),
    "no_halo": PLAIN.replace(M_h=0.0, n_steps=9),
    "one_step": PLAIN.replace(n_steps=1),
    # r^2 overflows float32 (and y is NaN) for one radius; the others share its launch
    "radius_out_of_float_range": PLAIN.replace(radii=np.array([5.0, 1e25, 80.0]), n_steps=40),
    "ragged_33": PLAIN.replace(n_q=3, n_mu=11, n_steps=65),
    "ragged_257": PLAIN.replace(n_q=257, n_mu=1, n_steps=64),
}


# masses below, at and between multiples of the group that an epilogue takes at a time
@pytest.mark.parametrize("n_mass", [3, 4, 5, 15])
@pytest.mark.parametrize("change", [{}, {"n_q": 257, "n_mu": 1}, {"n_q": 3, "n_mu": 11}])
def test_masses_of_a_small_launch_are_bitwise_the_counting_loop(n_mass, change):
    pb = PLAIN.replace(radii=np.geomspace(1.0, 3000.0, 5), n_steps=60,
                       masses=tuple(np.geomspace(0.01, 0.3, n_mass))).replace(**change)
    assert pb.n_out == 5 * n_mass
    for x, y in zip(*_both(pb, 256, 1)):
        assert np.array_equal(x, y)


# many radii of short runs: the launch is large enough for two trajectories a lane
LARGE = PLAIN.replace(radii=np.geomspace(1.0, 3000.0, 300), n_steps=40)


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("block,tpt", [(256, 1), (128, 3), (64, 3)])
def test_small_launch_is_bitwise_the_counting_loop(name, block, tpt):
    for a, b in zip(*_both(CASES[name], block, tpt)):
        assert np.array_equal(a, b, equal_nan=True)


# tiles of 64, 96 (three halves of a unit), 256, 288 and 1024 trajectories
@pytest.mark.parametrize("block,tpt", [(64, 1), (96, 1), (256, 1), (288, 1), (512, 2)])
@pytest.mark.parametrize("change", [{}, {"c": 25.0}, {"z_end": 6.0}, {"n_q": 257, "n_mu": 4}])
def test_large_launch_is_bitwise_the_counting_loop(change, block, tpt):
    for a, b in zip(*_both(LARGE.replace(**change), block, tpt)):
        assert np.array_equal(a, b, equal_nan=True)


# 3, 160 (one for an SM) and 480 tiles of 64 trajectories; odd shapes run whole tiles
@pytest.mark.parametrize("block,tpt", [(256, 1), (96, 1), (480, 1), (512, 2)])
@pytest.mark.parametrize("change", [{"n_q": 11, "n_mu": 5, "radii": np.array([2.0, 40.0, 900.0])}, {},
                                    {"radii": np.geomspace(1.0, 3000.0, 30)}, {"c": 25.0}])
def test_fp64_is_bitwise_the_counting_loop(change, block, tpt):
    pb = PLAIN.replace(precision=W.FP64, n_steps=20).replace(**change)
    for a, b in zip(*_both(pb, block, tpt)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("block,tpt", [(256, 1), (96, 1), (512, 2)])
def test_results_do_not_depend_on_what_shares_the_launch(block, tpt):
    """A small request alone (one trajectory a lane) and in a large batch (two)."""
    def results(problems):
        hs = [nu.create(pb, block=block, tpt=tpt) for pb in problems]
        b = nu.nu_batch_create(hs)
        try:
            nu.nu_batch_run(b)
            return [nu.nu_profile_result(h, pb.n_out) for h, pb in zip(hs, problems)]
        finally:
            nu.nu_batch_destroy(b)
            for h in hs:
                nu.nu_profile_destroy(h)

    small = PLAIN.replace(radii=np.array([3.0, 90.0]), n_q=37, n_mu=9, n_steps=100,
                          masses=(0.05, 0.1, 0.2))
    for a, b in zip(results([small])[0], results([LARGE, small])[1]):
        assert np.array_equal(a, b)


def test_interleaved_scans_give_the_results_of_fresh_tables():
    """More halos and cosmologies in turn than tables and backgrounds are kept: every
    result is that of the same request alone, and a handle's results outlive others'."""
    probs = [PLAIN.replace(M_h=m, Om=om, n_steps=n, radii=np.array([4.0, 60.0]), n_q=16, n_mu=8)
             for m in (1e12, 2e12, 4e12) for om in (0.29, 0.31, 0.33) for n in (50, 51)]
    first = [nu.profile(pb) for pb in probs]
    hs = [nu.create(pb) for pb in reversed(probs)]
    try:
        for h in hs:
            nu.nu_profile_run(h)
        again = [nu.nu_profile_result(h, 2) for h in hs][::-1]
    finally:
        for h in hs:
            nu.nu_profile_destroy(h)
    for a, b in zip(first, again):
        assert np.array_equal(a, b)
    assert len({r[0][0] for r in first}) == len(probs)


def test_results_beyond_the_host_block_are_copied():
    """Results of more values than the mapped host block holds, beside small ones."""
    big = PLAIN.replace(radii=np.geomspace(2000.0, 1e5, 70000), n_q=2, n_mu=1, n_steps=1)
    small = PLAIN.replace(n_steps=5)
    want = nu.profile(small)
    h = nu.create(big)
    try:
        nu.nu_profile_run(h)
        out, err = nu.nu_profile_result(h, big.n_out)
        assert np.array_equal(nu.profile(small), want)
        # beyond R every trajectory keeps its momentum
        assert np.allclose(out, 1.0, rtol=1e-6) and np.all(np.isfinite(err))
    finally:
        nu.nu_profile_destroy(h)
