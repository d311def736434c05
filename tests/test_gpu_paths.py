"""Sizes at which the kernels' tiles and dispatch rules can go wrong, against the oracle or the general path."""
import math

import numpy as np
import pytest
import torch
from scipy import special

import workloads as wl
from oracle import geometry as geo
from oracle import kernels as oker
from oracle import run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2507_05725_gb300 import fthms
    return fthms


@pytest.fixture(scope="module")
def ctx(F):
    torch.cuda.set_device(0)
    c = F.fthms_create(0, 0, None)
    yield c
    F.fthms_destroy(c)


def _rel(job, ref, problem):
    o = problem["options"]
    num = den = 0.0
    for m in range(1, o["M"] + 1):
        for j in range(len(problem["arcs"])):
            for q in range(o["Q"]):
                d = job.densities(j, m, q)
                for l in range(1, o["L"]):
                    r = ref.phi[(m, j, l)][q]
                    num += float(np.sum(np.abs(d[l] - r) ** 2))
                    den += float(np.sum(np.abs(r) ** 2))
    return math.sqrt(num / den)


@pytest.mark.parametrize("shift", [0, 1])
def test_densities_on_the_device_equal_the_host_copy(F, ctx, shift):
    """Byte for byte, also into a buffer that is only 8-byte aligned, for uneven N and several windows."""
    p = wl.random_small(5, n_curves=2, n_arcs_per_curve=2, Q=2, L=65, M=2)
    job = F.Job(ctx, p).run().wait()
    for j in range(4):
        for m in (0, 2):
            for q in range(2):
                want = F.fthms_densities(job.req, j, m, q)
                buf = torch.full((want.size + 2,), 7.0, dtype=torch.float64, device="cuda")
                torch.cuda.synchronize()
                F.fthms_densities_dev(job.req, j, m, q, buf.data_ptr() + 8 * shift, want.size)
                torch.cuda.synchronize()
                F.fthms_wait(job.req)
                F.fthms_stats(job.req)              # (a synchronising call on the job's stream)
                F.fthms_densities(job.req, j, m, q)
                got = buf.cpu().numpy()
                assert np.array_equal(got[shift:shift + want.size], want)
                assert got[shift + want.size] == 7.0 and (shift == 0 or got[0] == 7.0)
