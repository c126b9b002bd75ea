"""A C program that gives its handle back from an atexit handler it registered before
the library's first use, that is, after the library's own objects with static storage."""
import os
import subprocess

import pytest

from paper_2410_08267_gb300 import nuprof as nu

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include "nuprof.h"
static nu_profile* kept[3];
static void give_back(void)
{
    for (int i = 0; i < 3; ++i) nu_profile_destroy(kept[i]);
    fputs("given back\n", stderr);
}
int main(void)
{
    nu_cosmo cosmo = {0.31, 0.67, 1.95};
    nu_halo halo;
    nu_relic relic;
    nu_pgrid grid = {8, 4, 0.01, 10.0};
    nu_opts opts;
    double radii[2] = {10.0, 100.0}, out[2];
    atexit(give_back);
    memset(&halo, 0, sizeof halo);
    memset(&relic, 0, sizeof relic);
    memset(&opts, 0, sizeof opts);
    halo.M_h = 1e12;
    halo.c = 10.0;
    relic.m_eV = 0.1;
    opts.n_steps = 20;
    opts.precision = NU_MIXED;
    for (int i = 0; i < 3; ++i) {
        if (nu_profile_create(&cosmo, &halo, &relic, radii, 2, &grid, &opts, &kept[i])) return 2;
        if (nu_profile_run(kept[i], 0) || nu_profile_result(kept[i], out, 0, 2)) return 3;
    }
    return out[0] > 0.0 ? 0 : 4;
}
"""


def test_handles_given_back_while_the_process_exits(tmp_path):
    require_gpu()
    src, exe = tmp_path / "exit.c", tmp_path / "exit"
    src.write_text(SOURCE)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(nu.__file__))), "include")
    subprocess.run(["gcc", "-std=c99", "-I", include, str(src), "-o", str(exe), nu.LIB_PATH,
                    f"-Wl,-rpath,{os.path.dirname(nu.LIB_PATH)}"], check=True)
    # freed memory is overwritten, so that a use of it shows
    env = dict(os.environ, MALLOC_PERTURB_="165", GLIBC_TUNABLES="glibc.malloc.tcache_count=0")
    r = subprocess.run([str(exe)], env=env, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "given back" in r.stderr, (r.returncode, r.stderr)
