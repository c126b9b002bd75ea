"""The FP64 force's own arithmetic (the quotient y/(1+y), the series and the
logarithm of I(y)) through the force probe, where every factor but I(y) is known."""
import numpy as np
import pytest

from paper_2410_08267_gb300 import nuprof as nu
from paper_2410_08267_gb300 import workloads as W

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
PLAIN = W.plain_small(precision=W.FP64)[0]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


# y = r/r_s runs past the largest float (3.4e38) from c = 1e40 on
@pytest.mark.parametrize("c", [1e15, 1e30, 1e37, 1e38, 1e39, 1e60, 1e300])
def test_concentrations_beyond_the_float_range(c):
    pb = PLAIN.replace(c=c, n_steps=20, radii=np.array([5.0, 50.0, 500.0]))
    h = nu.create(pb)
    try:
        info = nu.nu_profile_info(h)
        r = np.geomspace(1e-3, 0.99, 200) * info["r200_kpc"]
        got = nu.nu_profile_force(h, 0, r)               # stage 0: z = 0
        y = r / info["r_s_kpc"]
        want = (np.log1p(y) - y / (1.0 + y)) / info["Ic"] / r ** 3 - info["R_kpc"] ** -3
        assert np.abs(got / want - 1.0).max() < 1e-14    # ~90 roundings, about 20 are made
        nu.nu_profile_run(h)
        out, err = nu.nu_profile_result(h, 3)
        assert np.all(np.isfinite(out)) and np.all(np.isfinite(err))
    finally:
        nu.nu_profile_destroy(h)
