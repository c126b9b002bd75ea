"""The kernels and tiles that plan_shape and whole_tiles choose give the bits of the
other paths at the sizes where a rule changes over, and what calls share in the host's
memory does not tie them to one another."""
import threading

import numpy as np
import pytest

from paper_2410_08267_gb300 import nuprof as nu
from paper_2410_08267_gb300 import workloads as W

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
PLAIN = W.plain_small(precision=W.MIXED)[0]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


# the sums of 256-trajectory tiles of 260 radii exceed the static array; tiles of 576
# and 960 trajectories end in a short pass, and 2^18 trajectories in a short tile
@pytest.mark.parametrize("block", [288, 480, 512])
def test_noalloc_wide_tiles_are_bitwise_the_handle_path(block):
    pb = PLAIN.replace(radii=np.geomspace(1.0, 3000.0, 260), n_q=1024, n_mu=256, n_steps=2)
    cosmo, halo, relic, radii, grid, opts = nu.structs(pb, torch_alloc=False, block=block, tpt=2)
    got = nu.nu_profile_compute_noalloc(cosmo, halo, relic, radii, grid, opts)
    want = nu.profile(pb, block=block, tpt=2)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


def _normal_and_counting(pb, grid=None):
    """n/nbar, error estimate and q_i of a run and of the counting launch."""
    h = nu.create(pb, flags=nu.NU_FLAG_KEEP_QI)
    b = nu.nu_batch_create([h])
    try:
        assert grid is None or nu.nu_batch_info(b)["grid"] == grid
        nu.nu_batch_run(b)
        runs = [(*nu.nu_profile_result(h, pb.n_out), nu.nu_profile_qi(h, pb.n_traj))]
        nu.nu_batch_branch_counts(b)
        runs.append((*nu.nu_profile_result(h, pb.n_out), nu.nu_profile_qi(h, pb.n_traj)))
        return runs
    finally:
        nu.nu_batch_destroy(b)
        nu.nu_profile_destroy(h)


# Tiles of 64 trajectories: up to one an SM (152), and up to 253 with three or more a
# radius, two pairs of warps share one, with one CTA an SM; otherwise a CTA takes one alone.
@pytest.mark.parametrize("n_q,n_mu,n_radii,grid", [(8, 16, 76, 152), (8, 16, 77, 154), (8, 16, 126, 252),
                                                   (8, 8, 153, 153), (12, 16, 51, 152), (12, 16, 84, 152),
                                                   (12, 16, 85, 255)])
def test_fp64_launches_around_the_split(n_q, n_mu, n_radii, grid):
    pb = PLAIN.replace(precision=W.FP64, n_steps=12, n_q=n_q, n_mu=n_mu,
                       radii=np.geomspace(1.0, 3000.0, n_radii))
    for x, y in zip(*_normal_and_counting(pb, grid)):
        assert np.array_equal(x, y)


# Mixed launches of 1024 trajectories a radius: one a lane in tiles of 128 (up to 4 CTAs
# on an SM) or two in tiles of 256 (6), by the most CTAs that an SM gets
@pytest.mark.parametrize("n_radii,grid", [(19, 152), (25, 200), (38, 304), (39, 312), (57, 456), (58, 232),
                                          (76, 304), (77, 608), (95, 608), (96, 384), (115, 608), (228, 608),
                                          (229, 912)])
def test_mixed_launches_around_the_rule(n_radii, grid):
    pb = PLAIN.replace(n_steps=20, n_q=32, n_mu=32, radii=np.geomspace(1.0, 3000.0, n_radii))
    for x, y in zip(*_normal_and_counting(pb, grid)):
        assert np.array_equal(x, y)


def test_fp64_results_do_not_depend_on_what_shares_the_launch():
    """A request alone (its pairs of points split over two warps), beside others of other
    series lengths, and the counting launch's: halos on both sides of y = 1 and beyond."""
    def q_i(problems, count):
        hs = [nu.create(pb, flags=nu.NU_FLAG_KEEP_QI) for pb in problems]
        b = nu.nu_batch_create(hs)
        try:
            nu.nu_batch_run(b)
            if count:
                nu.nu_batch_branch_counts(b)
            return [(nu.nu_profile_qi(h, pb.n_traj), *nu.nu_profile_result(h, pb.n_out))
                    for h, pb in zip(hs, problems)]
        finally:
            nu.nu_batch_destroy(b)
            for h in hs:
                nu.nu_profile_destroy(h)

    base = PLAIN.replace(precision=W.FP64, n_steps=60, n_q=37, n_mu=9)
    small = [base.replace(radii=np.array([0.01, 3.0, 90.0]), c=c, M_h=M)
             for c, M in ((0.9, 1e12), (4.0, 1e15), (10.0, 1e12), (40.0, 1e13))]
    beside = base.replace(radii=np.geomspace(0.1, 3000.0, 60), c=6.0)
    alone = [q_i([pb], False)[0] for pb in small]
    for together in (q_i([beside] + small, False)[1:], q_i(small[::-1], True)[::-1]):
        for one, other in zip(alone, together):
            for x, y in zip(one, other):
                assert np.array_equal(x, y)


# FP64 CTAs on an SM: the fewest that give each of its four schedulers a warp
@pytest.mark.parametrize("block,ctas", [(64, 2), (96, 2), (160, 1), (256, 2), (480, 1)])
def test_fp64_ctas_of_a_large_launch(block, ctas):
    pb = PLAIN.replace(precision=W.FP64, n_steps=2, radii=np.geomspace(1.0, 3000.0, 200))
    h = nu.create(pb, block=block)
    b = nu.nu_batch_create([h])
    try:
        assert nu.nu_batch_info(b)["grid"] == ctas * 152
    finally:
        nu.nu_batch_destroy(b)
        nu.nu_profile_destroy(h)


# Two trajectories a lane (the launch fills the chip), and warps that stay out of the NFW
# part for long: beyond R, grazing the shell, off the float range, without a halo.
@pytest.mark.parametrize("change", [{"radii": np.geomspace(1500.0, 30000.0, 300)},
                                    {"radii": np.geomspace(200.0, 1500.0, 300), "n_steps": 203},
                                    {"radii": np.append(np.geomspace(900.0, 3000.0, 299), 1e25)},
                                    {"radii": np.geomspace(900.0, 3000.0, 300), "c": 25.0, "z_end": 6.0},
                                    {"M_h": 0.0}])
def test_steps_outside_the_nfw_part_are_bitwise_the_counting_loop(change):
    pb = PLAIN.replace(radii=np.geomspace(1.0, 3000.0, 300), n_steps=120, n_q=40).replace(**change)
    for x, y in zip(*_normal_and_counting(pb)):
        assert np.array_equal(x, y, equal_nan=True)


def test_kept_tables_serve_both_precisions():
    """A halo's kept table, first made for a request of either mode, then read by the
    other, gives the results of a table made afresh."""
    mixed = PLAIN.replace(M_h=1.7e12, radii=np.array([4.0, 60.0]), n_q=16, n_mu=8, n_steps=50)
    both = [mixed, mixed.replace(precision=W.FP64)]
    fresh = {}
    for order in (both, both[::-1]):
        for k in range(9):                          # as many halos as tables are kept, and one
            nu.profile(mixed.replace(M_h=3e12 + 1e10 * k))
        for pb in order:
            got = nu.profile(pb)
            for a, b in zip(got, fresh.setdefault(int(pb.precision), got)):
                assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,n", [(W.MIXED, 8), (W.FP64, 5)])
def test_autotune_takes_shapes_of_one_tile_for_one_launch(precision, n):
    pb = PLAIN.replace(precision=precision, n_steps=20)
    h = nu.create(pb)
    try:
        r = nu.nu_autotune([h])
    finally:
        nu.nu_profile_destroy(h)
    by_tile = {}
    for block, tpt, flags, ms in r["candidates"]:
        by_tile.setdefault(block * min(tpt, 2), []).append((ms, block, tpt, flags))
    assert len(r["candidates"]) == n and set(by_tile) == {256, 384, 512}
    assert all(len({c[0] for c in same}) == 1 for same in by_tile.values())
    assert (r["best_ms"], r["block"], r["tpt"], r["flags"]) in [same[0] for same in by_tile.values()]


def test_requests_are_created_while_momenta_are_read():
    """Reading 6e7 momenta takes a tenth of a second or more; a request is created in
    some 50 us, in another thread, meanwhile."""
    pb = PLAIN.replace(radii=np.geomspace(1.0, 300.0, 60), n_q=2000, n_mu=512, n_steps=1)
    h = nu.create(pb, flags=nu.NU_FLAG_KEEP_QI)
    try:
        nu.nu_profile_run(h)
        nu.nu_profile_result(h, pb.n_out)
        reader = threading.Thread(target=nu.nu_profile_qi, args=(h, pb.n_traj))
        nu.nu_profile_destroy(nu.create(PLAIN))
        reader.start()
        created = 0
        while reader.is_alive():
            nu.nu_profile_destroy(nu.create(PLAIN))
            created += 1
        reader.join()
        assert created > 50
    finally:
        nu.nu_profile_destroy(h)
