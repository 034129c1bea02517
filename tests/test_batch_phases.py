"""The phase kernels of batches (explicit shapes): factorisation and sweeps."""
import dataclasses

import numpy as np
import pytest

from oracle import pf_oracle as O
from paper_1711_10579_gb300 import cases


@pytest.fixture(scope="module")
def env():
    from paper_1711_10579_gb300 import pf

    ctx = pf.pf_ctx_create(0)
    yield pf, ctx
    pf.pf_ctx_destroy(ctx)


def mesh(n):
    return cases.transmission_case(n, int(1.35 * n), max(n // 5, 1), 3, max_angle=0.06)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("S,B", [(2, 3), (4, 5), (8, 9), (16, 33), (32, 65)])
@pytest.mark.parametrize("n", [5, 33, 300])
def test_phase_kernels_match_oracle(env, n, S, B, prec):
    """Ragged batches in every scenarios-per-CTA shape: within 1e-6 of the
    oracle's solution, as every solve (the stop test's mismatch of 1e-8)."""
    pf, ctx = env
    case = mesh(n)
    pl, ql, pg = cases.scenario_loads(case, B, seed=5)
    c = pf.pf_create_case(ctx, case)
    try:
        o = pf.make_opts(precision=pf.PF_FP64 if prec == "fp64" else pf.PF_MIXED, scen_per_cta=S)
        vm, va, info = pf.pf_solve_batch(c, pl, ql, pg, o)
        assert np.all(info["status"] == 0) and np.all(info["mismatch"] <= 1e-8)
        for b in (0, B // 2, B - 1):
            r = O.newton_polar(case.with_loads(pl[b], ql[b], pg[b]))
            assert np.max(np.abs(vm[b] - r["vm"])) <= 1e-6
            assert np.max(np.abs(va[b] - r["va"])) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("S", [1, 2, 4, 8, 16])
def test_mixed_batch_in_a_large_power_base(env, S):
    """The same grid per unit of a power base 1e22 times larger: admittances and
    powers of 1e-22, whose 2x2 determinants are below the FP32 range.  The
    voltages are the oracle's in the ordinary base, within 1e-6."""
    pf, ctx = env
    case = mesh(33)
    k = 1e-22
    small = dataclasses.replace(case, br_r=case.br_r / k, br_x=case.br_x / k, br_b=case.br_b * k,
                                p_load=case.p_load * k, q_load=case.q_load * k,
                                p_gen=case.p_gen * k, q_gen=case.q_gen * k)
    B = 2 * S + 1
    pl, ql, pg = cases.scenario_loads(case, B, seed=5)
    c = pf.pf_create_case(ctx, small)
    try:
        o = pf.make_opts(precision=pf.PF_MIXED, scen_per_cta=S, tol=1e-8 * k)
        vm, va, info = pf.pf_solve_batch(c, pl * k, ql * k, pg * k, o)
        assert np.all(info["status"] == 0)
        for b in (0, B - 1):
            r = O.newton_polar(case.with_loads(pl[b], ql[b], pg[b]))
            assert np.max(np.abs(vm[b] - r["vm"])) <= 1e-6
            assert np.max(np.abs(va[b] - r["va"])) <= 1e-6
    finally:
        pf.pf_destroy_case(c)


@pytest.mark.gpu
@pytest.mark.parametrize("B", [305, 609, 2432])
def test_default_shape_of_mixed_batches(env, B):
    """Untuned mixed batches: about one CTA per SM, at most 8 scenarios each, and
    the bits of that shape asked for explicitly."""
    import torch

    pf, ctx = env
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    S = 1
    while S < 8 and B >= 2 * S * sms:
        S *= 2
    case = mesh(4000)
    pl, ql, pg = cases.scenario_loads(case, B, seed=7)
    c = pf.pf_create_case(ctx, case)
    try:
        assert pf.pf_launch_config(c, pf.make_opts(), B)["scen_per_cluster"] == S
        vm, va, info = pf.pf_solve_batch(c, pl, ql, pg, pf.make_opts())
        vm2, va2, info2 = pf.pf_solve_batch(c, pl, ql, pg, pf.make_opts(scen_per_cta=S))
        assert np.all(info["status"] == 0) and np.all(info2["status"] == 0)
        assert np.array_equal(vm, vm2) and np.array_equal(va, va2)
    finally:
        pf.pf_destroy_case(c)
