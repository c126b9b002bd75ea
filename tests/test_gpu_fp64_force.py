"""The FP64 force's own arithmetic (the quotient y/(1+y), the series and the
logarithm of I(y)) through the force probe, where every factor but I(y) is known."""
import ctypes
import ctypes.util
import math

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


def test_nfw_part_is_the_full_recurrence():
    """I(y) by the quotient y/(1+y) and the 51-term recurrence in plain FP64 (the C
    library's division and fma), over t = y/(1+y) from 1e-10 to 1.  At radii that are
    powers of two r, r^3 and the table's scale add no rounding; r^-1 is held to 2 ulp
    (five times in the product, 10u with u = 2^-53) and the rest rounds alike.  From
    y = 1 on I = log1p(y) - t: two libraries' logarithms, 1 ulp each, 4 times as large
    as their difference."""
    fma = ctypes.CDLL(ctypes.util.find_library("m")).fma
    fma.restype, fma.argtypes = ctypes.c_double, [ctypes.c_double] * 3
    r = 2.0 ** np.arange(-24, 8)
    seen = []
    for M in (1e12, 3e14):
        for c in np.geomspace(0.7, 60.0, 40):
            h = nu.create(PLAIN.replace(M_h=M, c=float(c), n_steps=1))
            try:
                info = nu.nu_profile_info(h)
                inside = r[r < 0.99 * info["r200_kpc"]]
                got = nu.nu_profile_force(h, 0, inside)
            finally:
                nu.nu_profile_destroy(h)
            S = 1.0 / info["r_s_kpc"]
            for ri, m in zip(inside, got):
                y = ri * S
                t = y / (1.0 + y)
                if t < 0.5:
                    p = 1.0 / 52
                    for k in range(49, -1, -1):
                        p = fma(p, t, 1.0 / (k + 2))
                    I = (t * t) * p
                else:
                    I = math.log1p(y) - t
                want = fma(I * (1.0 / info["Ic"]), ri ** -3, -1.0 / info["R_kpc"] ** 3)
                assert abs(m / want - 1.0) <= (2.0 ** -49 if t < 0.5 else 2.0 ** -48), (M, c, ri, t)
                seen.append(t)
    seen = np.array(seen)
    assert len(seen) > 2000 and seen.min() < 1e-9 and np.sum(seen >= 0.5) > 90
    assert np.all(np.histogram(seen, bins=[1e-9, 1e-6, 1e-3, 0.1, 0.2, 0.3, 0.36, 0.43, 0.5])[0] > 20)
