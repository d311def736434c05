"""Sizes at which the kernels' tiles and dispatch rules can go wrong, against the oracle or the general path."""
import copy
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


def _self_reference(curve, arc, N, kappa):
    """The oracle's self matrix with the log weights' phases k m pi/N reduced in integers (its own carry
    cos(k arccos t_i) with a rounding error that grows with k, 1e-12 of the largest entry at N = 1024)."""
    t, n = geo.cheb_nodes(N), np.arange(1, N)
    arc_ = geo.Arc(0, 0, curve, *arc)
    cosr = np.cos(np.arange(2 * N) * (np.pi / N))
    Fm = np.array([np.sum(cosr[(n * m) % (2 * N)] / n) for m in range(2 * N)])
    i = np.arange(N)
    rlog = -(np.pi / N) * (math.log(2.0) + Fm[np.abs(i[:, None] - i)] + Fm[i[:, None] + i + 1])
    X = arc_.point(t)[0]
    R = np.linalg.norm(X[:, None] - X[None], axis=-1)
    return oker.self_matrix(arc_, N, kappa) - special.j0(kappa * R) / (2.0 * np.pi) * (rlog - oker.rlog_self(N))


@pytest.mark.parametrize("N", [2, 3, 31, 32, 33, 64, 65, 1023, 1024])
def test_log_weights_at_block_edges(F, N):
    """The cosine sums F(0..N) come in blocks of 32 values; the matrix takes F(|i-l|) and F(i+l+1), folded at N.
    1e-13 of the largest entry: the bar of the self-matrix parity test."""
    curve, arc, kappa = wl.kite(0.1, 0.2), (-1.3, 1.1), 0.21 * N + 0.7
    A = torch.empty(2 * N * N, dtype=torch.float64, device="cuda")
    F.fthms_assemble_self(curve, arc, N, kappa, A.data_ptr())
    got = A.cpu().numpy().reshape(N, N, 2)
    got = (got[..., 0] + 1j * got[..., 1]).T
    ref = _self_reference(curve, arc, N, kappa)
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


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


@pytest.mark.parametrize("case", ["interpolated", "near-source", "few-nodes", "steep", "partitioned"])
def test_point_source_rows(F, ctx, case):
    """Incident data by interpolation in the distance from the source (many active nodes), node by node (source
    close to an arc, or few nodes) and sample by sample (a signal shorter than a run of samples)."""
    p = wl.config1(L=41, M=1, N=24 if case == "few-nodes" else 72)
    p["options"].update(H=4.0, n_period=256, W=16.0)
    if case == "near-source":
        p["signal"]["z0"] = [1.004, 0.0]
    if case == "steep":
        p["signal"].update(width=0.02, centre=1.5)
        p["options"]["n_period"] = 128
    ref = run_oracle(p)
    if case == "partitioned":
        p = copy.deepcopy(p)
        p["options"].update(omega_rank=1, omega_ranks=2)
        job = F.Job(ctx, p)
        job.set_allreduce(lambda buf, n, stream: None)
        job.run().wait()
        for j in range(3):
            for l, v in job.densities(j, 1, 0).items():
                assert np.linalg.norm(v - ref.phi[(1, j, l)][0]) <= 1e-11 * max(
                    np.linalg.norm(ref.phi[(1, j, k)][0]) for k in range(1, 41))
        return
    job = F.Job(ctx, p).run().wait()
    assert _rel(job, ref, p) < 1e-11


@pytest.mark.parametrize("Q", [1, 2, 3, 4])
@pytest.mark.parametrize("N,precision", [(31, 1), (33, 2), (0, 1), (0, 2)])
def test_every_step_rows_at_warp_and_band_edges(F, ctx, Q, N, precision):
    """Double-float cross rows evaluated every step (a warp per target row, 32 sources at a time, blocks of 1 to 8
    frequencies) against the FP64 form, stored rows: N around the warp width and bands of one to many equal-N
    frequencies, near rows on two curves.  1e-10: the mixed forms' bar."""
    p = wl.random_small(7, n_curves=2, n_arcs_per_curve=3, L=52, M=2, Q=Q, N_fixed=N, W=14.0, H=4.0, n_period=512)
    ref = F.Job(ctx, p).run().wait()
    p = copy.deepcopy(p)
    p["options"]["cross_mode"] = 1
    p["options"]["refine_max"] = 8
    job = F.Job(ctx, p, precision=precision).run().wait()
    num = den = 0.0
    for j in range(6):
        for q in range(Q):
            a, b = F.fthms_densities(ref.req, j, 2, q), F.fthms_densities(job.req, j, 2, q)
            num += float(np.sum((a - b) ** 2))
            den += float(np.sum(a ** 2))
    assert math.sqrt(num / den) < 1e-10
    t = ref.traces()
    assert np.max(np.abs(job.traces() - t)) < 1e-10 * np.max(np.abs(t))


@pytest.mark.parametrize("N", [5, 47, 96, 200])
@pytest.mark.parametrize("kappa", [0.01, 3.0, 19.9, 60.0, 700.0])
def test_self_matrix_over_the_hankel_ranges(F, N, kappa):
    """Taylor range, asymptotic range and both in one matrix, nearly closed arc (small |t - s| against R).  1e-13 of the
    largest entry, the bar of the self-matrix parity test."""
    curve, arc = wl.star(0.3, 5, 0.4), (0.1, 0.1 + 5.9)
    A = torch.empty(2 * N * N, dtype=torch.float64, device="cuda")
    F.fthms_assemble_self(curve, arc, N, kappa, A.data_ptr())
    got = A.cpu().numpy().reshape(N, N, 2)
    got = (got[..., 0] + 1j * got[..., 1]).T
    ref = _self_reference(curve, arc, N, kappa)
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("Q,N", [(1, 31), (1, 129), (2, 32), (2, 67), (3, 64), (4, 65)])
def test_stored_rows_in_fixed_point(F, ctx, precision, Q, N):
    """Stored cross rows (56-bit integers, carries every 32 sources, batches of 4 or 8) against rows evaluated every
    step in FP64: node counts around the batches and carries, an observation point next to the boundary (entries
    far above the others) and one far away.  1e-11 / 1e-10: the FP64 and mixed bars."""
    p = wl.random_small(11, n_curves=2, n_arcs_per_curve=3, L=40, M=2, Q=Q, N_fixed=N, W=12.0, H=4.0, n_period=512)
    p["options"]["obs"] = np.array([[0.0, 1.9], [40.0, -7.0], [9.0, 0.3]])
    p["options"]["refine_max"] = 8
    q_ = copy.deepcopy(p)
    q_["options"]["cross_mode"] = 1
    ref = F.Job(ctx, q_).run().wait()
    job = F.Job(ctx, p, precision=precision).run().wait()
    tol = 1e-11 if precision == 0 else 1e-10
    num = den = 0.0
    for j in range(6):
        for q in range(Q):
            a, b = F.fthms_densities(ref.req, j, 2, q), F.fthms_densities(job.req, j, 2, q)
            num += float(np.sum((a - b) ** 2))
            den += float(np.sum(a ** 2))
    assert math.sqrt(num / den) < tol
    t = ref.traces()
    assert np.all(np.abs(job.traces() - t) <= 10 * tol * np.max(np.abs(t), axis=1, keepdims=True))


def test_stored_rows_at_the_largest_node_count(F, ctx):
    """N = 1427 is the most that stored rows accept: the near tasks' shared memory is full there."""
    p = wl.random_small(2, n_arcs_per_curve=3, L=4, M=2, N_fixed=1427, W=24.0, H=0.3, n_period=64, kind=1)
    p["options"]["refine_max"] = 8
    jobs = []
    for mode in (0, 1):
        p["options"]["cross_mode"] = mode
        jobs.append(F.Job(ctx, p, precision=2).run())
        F.LIB.fthms_wait(jobs[-1].req, -1)
    for j in range(3):
        a, b = (F.fthms_densities(x.req, j, 2, 0) for x in jobs)
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("Q", [1, 2])
def test_fp64_fallback_with_rows_every_step(F, ctx, Q):
    """The FP64 re-run of a mixed job evaluates its rows over the same bands: bitwise the FP64 job's densities."""
    p = wl.random_small(7, n_curves=2, n_arcs_per_curve=3, L=52, M=2, Q=Q, N_fixed=33, W=14.0, H=4.0, n_period=512)
    p["options"]["cross_mode"] = 1
    ref = F.Job(ctx, p).run().wait()
    bad = copy.deepcopy(p)
    bad["options"].update(refine_tol=1e-30, refine_max=1, refine_fallback=1)
    job = F.Job(ctx, bad, precision=1).run().wait()
    assert job.stats()["fallback_runs"] == 1
    for j in range(6):
        for q in range(Q):
            assert np.array_equal(F.fthms_densities(ref.req, j, 2, q), F.fthms_densities(job.req, j, 2, q))


@pytest.mark.parametrize("n", [1, 63, 64, 65, 1000])
def test_bessel0_at_block_edges(F, n):
    """One value a thread in blocks of 64, nothing written past n.  5e-15 of the amplitude: scipy's own 3.4e-15 and
    the 1.5e-15 of the device functions."""
    z = np.exp(np.random.default_rng(n).uniform(np.log(1e-3), np.log(2000.0), n))
    zt = torch.tensor(z, dtype=torch.float64, device="cuda")
    out = [torch.full((n + 1,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
    F.fthms_bessel0(zt.data_ptr(), *(o.data_ptr() for o in out), n)
    torch.cuda.synchronize()
    assert all(float(o[n]) == 7.0 for o in out)
    j0, y0, yh = (o[:n].cpu().numpy() for o in out)
    rj, ry = special.j0(z), special.y0(z)
    amp = np.where(z > 1.0, np.sqrt(2.0 / (np.pi * z)), 1.0)
    assert np.max(np.abs(j0 - rj) / amp) < 5e-15
    assert np.max(np.abs(y0 - ry) / np.maximum(amp, np.abs(ry))) < 5e-15
    ryh = ry - (2.0 / np.pi) * (np.log(z / 2.0) + np.euler_gamma) * rj
    assert np.max((np.abs(yh - ryh) / (1.0 + np.abs(np.log(z))))[z < 20.0], initial=0.0) < 5e-15


def _in_units(p, s):
    """The same problem with lengths and times in units 1/s (s a power of two, so that every product is exact); the
    amplitude goes the other way, which keeps amplitude x time, the densities' unit."""
    p = copy.deepcopy(p)
    for c in p["curves"]:
        for k in ("ax", "bx", "ay", "by"):
            c[k] = [s * v for v in c[k]]
    g, o = p["signal"], p["options"]
    g.update(z0=[s * v for v in g["z0"]], carrier=g["carrier"] / s, centre=g["centre"] * s, width=g["width"] * s,
             amp=g["amp"] / s)
    o.update(W=o["W"] / s, H=o["H"] * s, obs=s * o["obs"], tout0=s * o["tout0"], dtout=s * o["dtout"])
    return p


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("bits", [-70, 70])
def test_results_do_not_depend_on_the_unit_of_length(F, ctx, precision, mode, bits):
    """Distances of 1e-21 and 1e21 (their squares leave FP32's range) with wavelengths to match: bit for bit the result
    in units of one, near and far rows, below and above z = 20."""
    p = wl.random_small(7, n_curves=2, n_arcs_per_curve=3, L=40, M=2, Q=2, W=14.0, H=4.0, n_period=512, kind=0)
    p["options"]["cross_mode"] = mode
    p["options"]["refine_max"] = 8
    s = 2.0 ** bits
    a, b = (F.Job(ctx, x, precision=precision).run().wait() for x in (p, _in_units(p, s)))
    assert np.array_equal(a.traces(), s * b.traces()) and np.max(np.abs(a.traces())) > 0.0
    for j in range(6):
        for q in range(2):
            assert np.array_equal(F.fthms_densities(a.req, j, 2, q), F.fthms_densities(b.req, j, 2, q))


@pytest.mark.parametrize("bits", [-480, -320, -80, 80, 480])
def test_self_matrix_does_not_depend_on_the_unit_of_length(F, bits):
    curve, arc, N, kappa, s = wl.star(0.3, 5, 0.4), (0.1, 2.2), 47, 19.9, 2.0 ** bits
    scaled = {k: [s * v for v in c] for k, c in curve.items()}
    out = []
    for c, k in ((curve, kappa), (scaled, kappa / s)):
        for call in (F.fthms_assemble_self, F.fthms_assemble_self_noalloc):
            A = torch.zeros(2 * N * N, dtype=torch.float64, device="cuda")
            call(c, arc, N, k, A.data_ptr())
            torch.cuda.synchronize()
            out.append(A.cpu())
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3]) and bool(torch.all(torch.isfinite(out[0])))


def test_stored_rows_of_many_large_sources(F, ctx):
    """A slice of rows over more sources than the FP64 form's limit counts (six arcs of 800 nodes, four windows): the mixed
    form takes it, the FP64 form and the fallback name the limit."""
    p = wl.random_small(7, n_curves=2, n_arcs_per_curve=3, L=3, M=2, Q=4, N_fixed=800, W=14.0, H=0.2, n_period=64, kind=1)
    p["options"]["refine_max"] = 8
    jobs = []
    for mode in (0, 1):
        p["options"]["cross_mode"] = mode
        jobs.append(F.Job(ctx, p, precision=2).run())
        F.LIB.fthms_wait(jobs[-1].req, -1)
    for j in range(6):
        for q in range(4):
            a, b = (F.fthms_densities(x.req, j, 2, q) for x in jobs)
            assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    t, u = (x.traces() for x in jobs)
    assert np.max(np.abs(t - u)) <= 1e-10 * np.max(np.abs(u)) and np.max(np.abs(u)) > 0.0
    p["options"].update(cross_mode=0, refine_tol=1e-30, refine_max=1, refine_fallback=1)
    with pytest.raises(F.FthmsError) as e:
        F.Job(ctx, p, precision=0)
    assert e.value.status == F.FTHMS_EINVAL and "232448" in str(e.value)
    job = F.Job(ctx, p, precision=2).run()
    with pytest.raises(F.FthmsError) as e:
        job.wait()
    assert e.value.status == F.FTHMS_ENOCONV and "limit" in str(e.value)


@pytest.mark.parametrize("N,L,signal,interpolated", [
    (72, 41, {}, True),
    (24, 41, {}, False),                                                          # few nodes
    (72, 41, dict(z0=[1.004, 0.0]), False),                                       # source next to an arc
    (160, 41, dict(z0=[1.2, 0.1], carrier=14.0, width=0.6, centre=3.0), False),   # samples and basis outgrow their memory
    (160, 97, dict(z0=[1.2, 0.1], carrier=14.0, width=0.6, centre=3.0), True),    # distances 0.2 to 2.2, high carrier
    (72, 97, dict(z0=[6.0, 1.0], carrier=14.0, width=0.6, centre=0.5), True)])    # distances 5.1 to 7.1
def test_point_source_rule(F, ctx, N, L, signal, interpolated):
    """Which jobs interpolate the incident field in the distance (two launches more: basis and product), and its accuracy
    where the distances differ most and the signal oscillates fastest.  1e-11: the FP64 bar."""
    p = wl.config1(L=L, M=1, N=N)
    p["options"].update(H=7.5 if signal.get("centre") == 0.5 else 4.0, n_period=256 if L < 50 else 512, W=16.0 if N < 100 else 24.0)
    p["signal"].update(signal)
    job = F.Job(ctx, p)
    F.fthms_profile(job.req, True)
    job.run().wait()
    assert F.fthms_stage_times(job.req)["incident"][1] == (4 if interpolated else 2)
    assert _rel(job, run_oracle(p), p) < 1e-11


@pytest.mark.parametrize("N", [8, 33, 96, 135])
def test_lu_thread_counts_give_the_same_factors(F, ctx, N):
    """FP64 jobs of systems up to 135 nodes factor with 128 threads a system, others with 256: the densities of small arcs are
    the same bit for bit with and without a large obstacle in the job (step 1 does not couple them)."""
    p = wl.random_small(9, n_arcs_per_curve=3, L=24, M=1, W=14.0, H=4.0, n_period=512, kind=1)
    p["curves"] = [wl.circle(1.0)]
    p["options"].update(N_min=N, N_off=0, N_ppw=N / (14.0 * 2.7))
    q = copy.deepcopy(p)
    q["curves"].append(wl.circle(20.0 if N < 33 else 3.0 if N > 60 else 6.0, 30.0, 0.0))
    q["arcs"] = q["arcs"] + [(1, a, b) for _, a, b in q["arcs"]]
    small, mixed = (F.Job(ctx, x).run().wait() for x in (p, q))
    assert {v.size for v in small.densities(0, 1, 0).values()} == {N}
    assert 135 < max(v.size for v in mixed.densities(3, 1, 0).values()) <= 800
    for j in range(3):
        assert np.array_equal(F.fthms_densities(small.req, j, 1, 0), F.fthms_densities(mixed.req, j, 1, 0))
