"""Resident solves (csrc/resident.cpp, csrc/resident.cu; feeders csrc/feeder.cpp,
csrc/feeder.cu): the host schedules executed on the CPU, and the kernels against the FP64 oracle at the sizes
where the cut into CTAs, the groups of 32 rows and the rounds have edges."""
import ctypes as C
import dataclasses
import os
import subprocess
import tempfile

import numpy as np
import pytest

from oracle import pf_oracle as O
from paper_1711_10579_gb300 import build, cases

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1711_10579_gb300", "csrc")


def mesh(n, seed=1):
    if n == 1:
        return dataclasses.replace(
            cases.two_bus_case(0.0, 0.0, 0.1, 0.1), n_bus=1, br_from=np.zeros(0, np.int32),
            br_to=np.zeros(0, np.int32), br_r=np.zeros(0), br_x=np.zeros(0), br_b=np.zeros(0),
            **{k: getattr(cases.two_bus_case(0.0, 0.0, 0.1, 0.1), k)[:1] for k in
               ("bus_type", "v_set", "p_gen", "q_gen", "p_load", "q_load", "zip")})
    if n == 2:
        return cases.two_bus_case(0.9, 0.3, 0.02, 0.15)
    m = max(n - 1, int(1.35 * n)) if n > 4 else n - 1
    return cases.transmission_case(n, m, max(1, n // 5), seed, max_angle=0.06)


# ----------------------------------------------------------------------------
# the schedule, on the CPU
# ----------------------------------------------------------------------------

@pytest.fixture(scope="module")
def host():
    so = os.path.join(tempfile.mkdtemp(prefix="resident"), "resident_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                           "-I", os.path.join(build._cuda_home(), "include"), "-o", so,
                           os.path.join(HERE, "resident_host.cpp"),
                           *[os.path.join(CSRC, f) for f in
                             ("resident.cpp", "feeder.cpp", "symbolic.cpp")]])
    return C.CDLL(so)


@pytest.mark.parametrize("P,threads", [(1, 32), (1, 512), (2, 64), (4, 128), (16, 512)])
@pytest.mark.parametrize("n", [1, 2, 3, 14, 33, 300, 2000])
def test_schedule_solves_the_system(host, n, P, threads):
    """Residuals of a diagonally dominant random system in FP64: a few ulps of
    the entries times the row length."""
    g = mesh(n)
    f, t = (np.ascontiguousarray(a, np.int32) for a in (g.br_from, g.br_to))
    err, parts = C.c_double(-1.0), C.c_int(0)
    rc = host.resident_check(n, len(f), f.ctypes.data_as(C.c_void_p), t.ctypes.data_as(C.c_void_p),
                             P, threads, 0, C.byref(err), C.byref(parts))
    assert rc == 0
    assert 0.0 <= err.value <= 1e-13
    if n == 2000 and P > 1:
        assert parts.value == P + 1  # every CTA has its own subtrees, and there is a top


def test_schedule_of_a_tree_and_of_a_star(host):
    feeder = cases.feeder_case(700, 3)
    star = (np.zeros(299, np.int32), np.arange(1, 300, dtype=np.int32))
    for f, t, n in ((feeder.br_from, feeder.br_to, 700), (*star, 300)):
        f, t = (np.ascontiguousarray(a, np.int32) for a in (f, t))
        for P in (1, 4):
            err, parts = C.c_double(-1.0), C.c_int(0)
            assert host.resident_check(n, len(f), f.ctypes.data_as(C.c_void_p),
                                       t.ctypes.data_as(C.c_void_p), P, 128, 0, C.byref(err),
                                       C.byref(parts)) == 0
            assert 0.0 <= err.value <= 1e-13


@pytest.mark.parametrize("n", [1, 2, 14, 33, 300])
def test_schedule_of_an_incomplete_factor(host, n):
    g = mesh(n)
    f, t = (np.ascontiguousarray(a, np.int32) for a in (g.br_from, g.br_to))
    err, parts = C.c_double(-1.0), C.c_int(0)
    assert host.resident_check(n, len(f), f.ctypes.data_as(C.c_void_p), t.ctypes.data_as(C.c_void_p),
                               1, 64, 1, C.byref(err), C.byref(parts)) == 0
    assert 0.0 <= err.value <= 1e-14


@pytest.mark.parametrize("P,groups", [(1, 4), (1, 32), (2, 8), (4, 16), (16, 32)])
@pytest.mark.parametrize("n", [1, 2, 40, 700, 3000])
def test_feeder_schedule_solves_the_system(host, n, P, groups):
    """Scalar stand-ins for the 6x6 blocks; a feeder too small for P parts has
    no plan (the other kernels solve it)."""
    g = cases.feeder_case(n, 4) if n > 1 else None
    f, t = ((np.ascontiguousarray(a, np.int32) for a in (g.br_from, g.br_to)) if g is not None
            else (np.zeros(0, np.int32),) * 2)
    kinds = np.array([7], np.int8) if g is None else g.phases.astype(np.int8)
    kinds[0] |= 8
    err, levels = C.c_double(-1.0), C.c_int(0)
    rc = host.feeder_check(n, *[a.ctypes.data_as(C.c_void_p) for a in (f, t, kinds)], P, groups,
                           C.byref(err), C.byref(levels))
    if P > 1 and n < 40 * P and rc == 100:
        return  # no plan
    assert rc == 0
    assert 0.0 <= err.value <= 1e-13


def test_feeder_schedule_refuses_pv_nodes(host):
    g = cases.feeder_case(40, 1)
    f, t = (np.ascontiguousarray(a, np.int32) for a in (g.br_from, g.br_to))
    kinds = g.phases.astype(np.int8)
    kinds[5] |= 16
    err, levels = C.c_double(), C.c_int()
    args = lambda: [a.ctypes.data_as(C.c_void_p) for a in (f, t, kinds)]
    assert host.feeder_check(40, *args(), 1, 8, C.byref(err), C.byref(levels)) == 100


def test_analysis_of_a_comb_is_quick():
    """A corridor of 10,000 buses with a bus at each (0.06 s; a cut that packs its
    parts anew for every bus of the corridor takes seconds)."""
    import time

    from paper_1711_10579_gb300 import pf

    n, h = 20_000, 10_000
    one = cases.two_bus_case(0.0, 0.0, 0.1, 0.1)
    f = np.r_[np.arange(h - 1), np.arange(h)].astype(np.int32)
    t = np.r_[np.arange(1, h), np.arange(h, n)].astype(np.int32)
    z = np.zeros(n)
    case = dataclasses.replace(one, n_bus=n, br_from=f, br_to=t, br_r=np.full(n - 1, 0.01),
                               br_x=np.full(n - 1, 0.1), br_b=np.zeros(n - 1),
                               bus_type=np.r_[0, np.full(n - 1, 2)].astype(np.int32), v_set=z + 1.0,
                               p_gen=z, q_gen=z, p_load=z, q_load=z,
                               zip=np.tile([1.0, 0.0, 0.0], (n, 1)))
    t0 = time.perf_counter()
    assert pf.pf_analyze(case)["n_bus"] == n
    assert time.perf_counter() - t0 < 1.5


# ----------------------------------------------------------------------------
# the kernels
# ----------------------------------------------------------------------------

@pytest.fixture(scope="module")
def env():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1711_10579_gb300 import pf

    ctx = pf.pf_ctx_create(0)
    yield pf, ctx
    pf.pf_ctx_destroy(ctx)


def _loads(case, B, seed):
    if case.n_bus <= 2:
        s = np.linspace(1.0, 0.5, B)[:, None]
        return case.p_load[None] * s, case.q_load[None] * s, np.repeat(case.p_gen[None], B, 0)
    return cases.scenario_loads(case, B, seed=seed)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,P", [(1, 1), (2, 1), (3, 2), (14, 1), (31, 1), (33, 4), (129, 2), (500, 1),
                                 (500, 16), (2000, 8)])
def test_resident_matches_oracle(env, n, P, prec):
    """Single solves and a ragged batch on P CTAs, ZIP loads and a PQ bus with
    generation among them, with and without FP64 refinement: within 1e-6 of
    the oracle's solution, as every solve (the stop test's mismatch of 1e-8)."""
    pf, ctx = env
    case = mesh(n)
    if n > 2:
        zipf = np.tile([1.0, 0.0, 0.0], (n, 1))
        zipf[1::2] = [0.4, 0.35, 0.25]
        qg = np.zeros(n)
        qg[np.flatnonzero(case.bus_type == cases.PQ)[0]] = 1e-3
        case = dataclasses.replace(case, zip=zipf, q_gen=qg)
    pl, ql, pg = _loads(case, 3, seed=5)
    refs = [O.newton_polar(case.with_loads(pl[b], ql[b], pg[b])) if n > 1 else
            {"vm": case.v_set, "va": np.zeros(1)} for b in range(3)]
    c = pf.pf_create_case(ctx, case)
    try:
        for rs in (0.1, 0.0):
            o = pf.make_opts(precision=pf.PF_FP64 if prec == "fp64" else pf.PF_MIXED,
                             cluster_size=P, refine_stall=rs)
            shape = pf.pf_launch_config(c, o, 3)
            assert shape["cluster"] == P and shape["grid"] == 3 * P
            vm, va, info = pf.pf_solve_batch(c, pl, ql, pg, o)
            vm1, va1, info1 = pf.pf_solve_batch(c, pl[:1], ql[:1], pg[:1], o)
            assert np.all(info["status"] == 0) and np.all(info["mismatch"] <= 1e-8)
            # the same launch shape: the scenario alone is the same bit for bit
            assert np.array_equal(vm[0], vm1[0]) and np.array_equal(va[0], va1[0])
            assert np.all(info["linear_iterations"] >= info["iterations"])
            for b, r in enumerate(refs):
                assert np.max(np.abs(vm[b] - r["vm"])) <= 1e-6
                assert np.max(np.abs(va[b] - r["va"])) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,B", [(14, 153), (14, 1217), (14, 9728), (60, 305), (300, 153), (300, 609), (500, 305),
                                 (500, 609)])
def test_resident_batch_threads(env, n, B, prec):
    """The threads of a CTA follow the batch: every shape of a scenario's CTA
    gives the same bits (the order of a block's updates is the plan's)."""
    pf, ctx = env
    case = mesh(n)
    pl, ql, pg = _loads(case, B, seed=9)
    c = pf.pf_create_case(ctx, case)
    try:
        o = pf.make_opts(precision=pf.PF_FP64 if prec == "fp64" else pf.PF_MIXED, cluster_size=1)
        assert pf.pf_launch_config(c, o, B)["threads"] <= pf.pf_launch_config(c, o, 3)["threads"]
        vm, va, info = pf.pf_solve_batch(c, pl, ql, pg, o)
        assert np.all(info["status"] == 0)
        for k in (0, B // 2, B - 3):
            vm3, va3, _ = pf.pf_solve_batch(c, pl[k:k + 3], ql[k:k + 3], pg[k:k + 3], o)
            assert np.array_equal(vm[k:k + 3], vm3) and np.array_equal(va[k:k + 3], va3)
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n", [("mesh", 33), ("mesh", 500), ("mesh", 3906), ("feeder", 1106)])
def test_mixed_solves_keep_their_kernels(env, kind, n):
    """Mixed solves of more than 32 buses or 1,000 nodes: alone, in a batch, served
    and under reactive limits the bits of the persistent and the phase kernels
    (explicit threads), whose FP32 sums are in another order than the resident
    kernels'."""
    pf, ctx = env
    B = 4
    if kind == "mesh":
        case = cases.with_q_limits(mesh(n), 2)
        loads = cases.scenario_loads(case, B, seed=3)
        full = 512
    else:
        case = cases.feeder_case(n, 43)
        loads = (*[a.reshape(B, -1) for a in cases.feeder_scenario_loads(case, B, seed=3)], None)
        full = 256
    one = [None if a is None else a[:1] for a in loads]
    row = [None if a is None else a[0] for a in loads]
    c = pf.pf_create_case(ctx, case)
    try:
        def same(x, y):
            assert np.all(x[2]["status"] == 0) and np.all(y[2]["status"] == 0)
            assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])

        alone = pf.pf_solve_batch(c, *one, pf.make_opts())
        same(alone, pf.pf_solve_batch(c, *one, pf.make_opts(block_threads=full)))
        same(pf.pf_solve(c, pf.make_opts()), pf.pf_solve(c, pf.make_opts(block_threads=full)))
        same(pf.pf_solve_batch(c, *loads, pf.make_opts()),
             pf.pf_solve_batch(c, *loads, pf.make_opts(scen_per_cta=1)))
        t = pf.pf_submit(ctx, c, *row, pf.make_opts())
        pf.pf_drain(ctx)
        vm, va, info = pf.pf_poll(ctx, t, c.slots)
        same((vm, va, info), (alone[0][0], alone[1][0], {"status": alone[2]["status"][0]}))
        if kind == "mesh":
            limited = pf.pf_solve_batch(c, *one, pf.make_opts(q_limits=1))
            same(limited, pf.pf_solve_batch(c, *one, pf.make_opts(q_limits=1, block_threads=full)))
            t = pf.pf_submit(ctx, c, *row, pf.make_opts(q_limits=1))
            pf.pf_drain(ctx)
            vm, va, info = pf.pf_poll(ctx, t, c.slots)
            same((vm, va, info), (limited[0][0], limited[1][0], {"status": limited[2]["status"][0]}))
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
def test_resident_reports_failures(env):
    """A scenario past the loading nose next to one that converges, and an
    iteration limit."""
    pf, ctx = env
    case = cases.two_bus_case(50.0, 20.0, 0.02, 0.15)
    c = pf.pf_create_case(ctx, case)
    pl = np.array([[0.0, 50.0], [0.0, 0.9]])
    ql = np.array([[0.0, 20.0], [0.0, 0.3]])
    _, _, info = pf.pf_solve_batch(c, pl, ql, None, pf.make_opts(max_iter=20))
    assert info["status"][0] in (pf.PF_ERR_MAXITER, pf.PF_ERR_DIVERGED, pf.PF_ERR_SINGULAR)
    assert info["status"][1] == 0
    _, _, info = pf.pf_solve_batch(c, pl, ql, None, pf.make_opts(max_iter=0))
    assert np.all(info["status"] == pf.PF_ERR_MAXITER) and np.all(info["iterations"] == 0)
    pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,P", [(1, 1), (2, 1), (11, 1), (33, 1), (300, 2), (300, 4), (1000, 4),
                                 (1000, 16)])
def test_resident_feeder_matches_oracle(env, n, P, prec):
    """Feeders on P CTAs, alone and in a ragged batch, with and without FP64
    refinement: within 1e-6 of the oracle's solution (the stop test's mismatch
    of 1e-8); a scenario alone equals the same in a batch bit for bit."""
    pf, ctx = env
    if n == 1:
        z = np.zeros((1, 3))
        case = cases.ThreePhaseCase(1, 0, np.array([7], np.uint8), z, z, np.array([[0.5, 0.3, 0.2]]),
                                    np.zeros(0, np.int32), np.zeros(0, np.int32),
                                    np.zeros(0, np.uint8), np.zeros((0, 3, 3), complex))
    else:
        case = cases.feeder_case(n, 5)
    pl, ql = cases.feeder_scenario_loads(case, 3, seed=2)
    refs = [O.newton_cim(case.with_loads(pl[b], ql[b]))["V"] if n > 1 else
            O.cim_flat_start(case) for b in range(3)]
    c = pf.pf_create_case(ctx, case)
    try:
        for rs in (0.1, 0.0):
            o = pf.make_opts(precision=pf.PF_FP64 if prec == "fp64" else pf.PF_MIXED,
                             cluster_size=P, refine_stall=rs)
            shape = pf.pf_launch_config(c, o, 3)
            assert shape["cluster"] == P and shape["grid"] == 3 * P
            vm, va, info = pf.pf_solve_batch(c, pl.reshape(3, -1), ql.reshape(3, -1), None, o)
            vm1, va1, _ = pf.pf_solve_batch(c, pl[:1].reshape(1, -1), ql[:1].reshape(1, -1), None, o)
            assert np.all(info["status"] == 0) and np.all(info["mismatch"] <= 1e-8)
            assert np.array_equal(vm[0], vm1[0]) and np.array_equal(va[0], va1[0])
            for b, V in enumerate(refs):
                V = V.reshape(-1)
                assert np.max(np.abs(vm[b] * np.exp(1j * va[b]) - V)) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,P", [(2, 2), (3, 2), (11, 4), (40, 2), (40, 4), (40, 16), (100, 16)])
def test_small_feeders_on_clusters(env, n, P, prec):
    """Parts of a node or none: the oracle's solution, on the plan or, where there is
    none, on the other kernels."""
    pf, ctx = env
    case = cases.feeder_case(n, 5)
    V = O.newton_cim(case)["V"].reshape(-1)
    c = pf.pf_create_case(ctx, case)
    try:
        o = pf.make_opts(precision=prec, cluster_size=P)
        shape = pf.pf_launch_config(c, o, 1)
        assert shape["cluster"] == P
        vm, va, info = pf.pf_solve(c, o)
        assert info["status"] == 0
        assert np.max(np.abs(vm * np.exp(1j * va) - V)) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("n,m", [(2, 30), (14, 30), (33, 7), (300, 30), (1000, 5), (1000, 40)])
def test_resident_krylov_matches_oracle(env, n, m):
    """GMRES(m) with ILU(0), restarted and not, alone and in a ragged batch."""
    pf, ctx = env
    case = mesh(n)
    pl, ql, pg = _loads(case, 3, seed=9)
    c = pf.pf_create_case(ctx, case)
    try:
        o = pf.make_opts(method=pf.PF_NK, precision=pf.PF_FP64, gmres_restart=m, nk_fallback=0, gmres_max_iter=2000)
        assert pf.pf_launch_config(c, o, 3)["grid"] == 3
        vm, va, info = pf.pf_solve_batch(c, pl, ql, pg, o)
        vm1, va1, info1 = pf.pf_solve_batch(c, pl[:1], ql[:1], pg[:1], o)
        assert np.all(info["status"] == 0) and np.all(info["mismatch"] <= 1e-8)
        assert np.all(info["linear_iterations"] >= info["iterations"])
        assert np.array_equal(vm[0], vm1[0]) and np.array_equal(va[0], va1[0])
        for b in range(3):
            r = O.newton_polar(case.with_loads(pl[b], ql[b], pg[b]))
            assert np.max(np.abs(vm[b] - r["vm"])) <= 1e-6
            assert np.max(np.abs(va[b] - r["va"])) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind,n,P,B", [("mesh", 500, 16, 3000), ("mesh", 2000, 4, 2000),
                                        ("feeder", 1000, 16, 500)])
def test_asked_ctas_keep_the_batch_rule(env, kind, n, P, B, prec):
    """CTAs per scenario asked for: resident in a small batch; a batch too large for
    resident solves runs as without them."""
    pf, ctx = env
    c = pf.pf_create_case(ctx, mesh(n) if kind == "mesh" else cases.feeder_case(n, 5))
    try:
        o, plain = (pf.make_opts(precision=prec, cluster_size=q) for q in (P, 0))
        small = pf.pf_launch_config(c, o, 3)
        assert small["cluster"] == P and small["grid"] == 3 * P
        assert pf.pf_launch_config(c, o, B)["cluster"] == 1
        assert pf.pf_launch_config(c, o, B) == pf.pf_launch_config(c, plain, B)
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("method,prec,n,B", [("nk", 0, 60, 40), ("nk", 1, 60, 40), ("nr", 0, 300, 64),
                                             ("nr", 1, 300, 64)])
def test_tuned_choice_is_what_runs(env, method, prec, n, B):
    """After pf_autotune the launch is the returned shape, or the resident solves
    where it returned none; CTAs per scenario asked for come before it."""
    pf, ctx = env
    c = pf.pf_create_case(ctx, mesh(n))
    m = pf.PF_NK if method == "nk" else pf.PF_NR
    try:
        got = pf.pf_autotune(c, B, pf.make_opts(method=m, precision=prec, nk_fallback=0))
        shape = pf.pf_launch_config(c, pf.make_opts(method=m, precision=prec), B)
        if got.scen_per_cta:
            assert shape["scen_per_cluster"] == got.scen_per_cta
            assert shape["threads"] == got.block_threads
        else:
            assert shape["scen_per_cluster"] == 1 and shape["grid"] == B * shape["cluster"]
            assert got.block_threads == 0
        if method == "nr":
            asked = pf.pf_launch_config(c, pf.make_opts(method=m, precision=prec, cluster_size=2), B)
            assert asked["cluster"] == 2 and asked["grid"] == 2 * B
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind,n,P", [("mesh", 2, 0), ("mesh", 14, 0), ("mesh", 32, 0), ("mesh", 33, 0),
                                      ("mesh", 500, 4), ("feeder", 40, 0), ("feeder", 300, 0)])
def test_solves_in_a_large_power_base(env, kind, n, P, prec):
    """The same grid per unit of a power base 1e22 times larger: admittances and
    powers of 1e-22, whose 2x2 determinants are below the FP32 range.  Within
    1e-6 of the oracle's voltages in the ordinary base."""
    pf, ctx = env
    k = 1e-22
    if kind == "mesh":
        case = mesh(n)
        ref = O.newton_polar(case)
        ref = ref["vm"] * np.exp(1j * ref["va"])
        small = dataclasses.replace(case, br_r=case.br_r / k, br_x=case.br_x / k, br_b=case.br_b * k,
                                    p_load=case.p_load * k, q_load=case.q_load * k,
                                    p_gen=case.p_gen * k, q_gen=case.q_gen * k)
    else:
        case = cases.feeder_case(n, 5)
        ref = O.newton_cim(case)["V"].reshape(-1)
        small = dataclasses.replace(case, br_z=case.br_z / k, p_load=case.p_load * k,
                                    q_load=case.q_load * k)
    c = pf.pf_create_case(ctx, small)
    try:
        vm, va, info = pf.pf_solve(c, pf.make_opts(precision=prec, cluster_size=P, tol=1e-8 * k))
        assert info["status"] == 0
        on = np.abs(ref) > 0
        assert np.max(np.abs(vm * np.exp(1j * va) - ref)[on]) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n", [("mesh", 1), ("mesh", 14), ("mesh", 33), ("mesh", 2749), ("mesh", 10000),
                                    ("feeder", 40), ("feeder", 1106), ("feeder", 8000)])
def test_analysis_counts_what_a_case_holds(env, kind, n):
    """pf_analyze, which needs no GPU, against the created case; asking for a launch
    configuration uploads nothing, the batch itself does."""
    pf, ctx = env
    case = mesh(n) if kind == "mesh" else cases.feeder_case(n, 3)
    c = pf.pf_create_case(ctx, case)
    try:
        held = lambda: pf.pf_case_get_stats(c)["device_bytes"]
        created = held()
        assert pf.pf_analyze(case)["device_bytes"] == created
        o = pf.make_opts(precision=pf.PF_FP64)
        shape = pf.pf_launch_config(c, o, 3)
        assert held() == created
        if n == 2749:  # a batch runs on fewer CTAs than one solve: another plan
            assert shape["cluster"] > 1 and shape["scen_per_cluster"] == 1
            pl, ql, pg = _loads(case, 3, seed=1)
            assert np.all(pf.pf_solve_batch(c, pl, ql, pg, o)[2]["status"] == 0)
            assert held() > created
            assert pf.pf_launch_config(c, o, 3) == shape
    finally:
        pf.pf_destroy_case(c)
